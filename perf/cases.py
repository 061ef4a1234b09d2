"""What a user of the package has it do, as cases a timing program can prepare, run and check.

Every case goes through the public entry points of ``paper_2212_06985_gb300``.  Inputs are made
on the GPU from a seed: the simulator's own noise (keyed by the run's seed), or bits drawn with a
seeded torch generator where a caller brings measured syndromes.
"""
from __future__ import annotations

import functools
import math
import os

import numpy as np
import torch

import paper_2212_06985_gb300 as t3d

DEV = "cuda:0"


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # The smallest whole run: plain flip on the L = 4 code, 10^4 samples, 32 applications a
        # cycle, four noisy cycles and a noiseless round -- about 170 tiny steps, so latency counts.
        dict(name="flip run L4", kind="run", L=4, samples=10_000, T=4, p=0.01, schedule="F", n_apply=32,
             perfect=32),
        # A control loop's single steps on a small ragged batch (the last word is partly filled):
        # noise, measurement, FFPFF and the readout as separate calls.
        dict(name="steps L8", kind="steps", L=8, samples=1_000, p=0.03, schedule="FFPFF", n_apply=5),
        # A point of a threshold curve: the whole T = L run of the p-flip decoder, 10^6 samples.
        dict(name="pflip run L8", kind="run", L=8, samples=1_000_000, T=8, p=0.03, schedule="FFPFF", n_apply=5,
             perfect=0),
        # The flip / p-flip throughput workload: one code cycle of 10^5 samples at L = 32.
        dict(name="pflip cycle L32", kind="batch", L=32, L2=0, samples=100_000, p=0.04, decoder="pflip", bp_iters=0,
             schedule="FFPFF", n_apply=5),
        # The headline workload, BP with 16 iterations and 32 applications of PFFPFF at L = 32, in a
        # batch that leaves room for three of them on the card.
        dict(name="bp cycle L32", kind="batch", L=32, L2=0, samples=12_500, p=0.04, decoder="bp", bp_iters=16,
             schedule="PFFPFF", n_apply=32),
        # The same decoder on two lattice sizes in shared launches.
        dict(name="bp cycle L16+24", kind="batch", L=16, L2=24, samples=10_000, p=0.04, decoder="bp", bp_iters=16,
             schedule="PFFPFF", n_apply=32),
        # A threshold run of p-BP (20 iterations, then PFFPFF) at the paper's smallest size, captured
        # in a CUDA graph, from a fresh code.
        dict(name="pbp graph L14", kind="graph", L=14, samples=3_000, T=6, p=0.06, bp_iters=20, schedule="PFFPFF",
             n_apply=6),
        # The learned pre-decoder ahead of the schedule with its BP fallback.
        dict(name="learned cycle L24", kind="batch", L=24, L2=0, samples=20_000, p=0.04, decoder="learned", bp_iters=16,
             schedule="PFFPFF", n_apply=32),
        # One training step of the pre-decoder as it is trained: L = 12, 2,048 codes.
        dict(name="train L12", kind="train", L=12, samples=2_048, p=0.04),
        # One BP decode of a caller's measured syndromes with the posteriors read out, the cube
        # meta-checks on (an odd lattice size of the threshold sets, a ragged batch).
        dict(name="meta bp L18", kind="bp", L=18, samples=1_500, p=0.04, bp_iters=12, meta=True),
        # Another LDPC code: the Z checks of a hypergraph product, 62,500 qubits; noise, measurement,
        # BP with posteriors, then the flip / p-flip schedule.
        dict(name="hgp code", kind="tanner", classical=200, samples=2_000, p=0.015, bp_iters=20, schedule="PFFPFF",
             n_apply=6),
        # Syndromes that arrive as bytes, one sample a row: packed, decoded by flip until they
        # clear, and the corrections and what is left of the syndromes handed back as bytes.
        dict(name="bytes L12", kind="bits", L=12, samples=20_000, p=0.01, sweeps=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "steps", "cycle", "cycle", "bp cycle", "bp cycle", "graph", "learned", "train", "bp",
                       "tanner", "bits"])
    p = round(rng.uniform(0.01, 0.045), 4)
    if kind == "run":
        L = rng.randint(3, 16)
        room = 400_000_000 // (3 * L ** 3)
        return dict(kind="run", L=L, samples=_log(rng, 500, min(1_000_000, room)), T=rng.randint(2, 8), p=p,
                    schedule=rng.choice(["F", "FFPFF", "FFF"]), n_apply=rng.randint(1, 9),
                    perfect=rng.choice([0, 32]))
    if kind == "steps":
        return dict(kind="steps", L=rng.randint(3, 16), samples=_log(rng, 40, 20_000), p=p,
                    schedule=rng.choice(["FFPFF", "PFFPFF"]), n_apply=rng.randint(1, 9))
    if kind == "cycle":
        L = rng.randint(8, 48)
        room = 6_000_000_000 // (3 * L ** 3)
        return dict(kind="batch", L=L, L2=0, samples=_log(rng, 1_000, min(100_000, room)), p=p, decoder="pflip",
                    bp_iters=0, schedule=rng.choice(["FFPFF", "FFFPFFFPF"]), n_apply=rng.randint(1, 9))
    if kind == "bp cycle":
        L, L2 = rng.randint(8, 40), rng.choice([0, 0, 14, 18, 24])
        room = 1_000_000_000 // (3 * L ** 3 + 3 * L2 ** 3)
        return dict(kind="batch", L=L, L2=L2, samples=_log(rng, 300, min(50_000, room)), p=p, decoder="bp",
                    bp_iters=rng.choice([8, 16]), schedule="PFFPFF", n_apply=rng.choice([6, 32]))
    if kind == "graph":
        return dict(kind="graph", L=rng.choice([9, 14, 18]), samples=_log(rng, 300, 3_000), T=rng.randint(2, 5),
                    p=round(rng.uniform(0.03, 0.06), 4), bp_iters=rng.choice([10, 20]), schedule="PFFPFF", n_apply=6)
    if kind == "learned":
        L = rng.randint(8, 24)
        room = 800_000_000 // (3 * L ** 3)
        return dict(kind="batch", L=L, L2=0, samples=_log(rng, 500, min(50_000, room)), p=p, decoder="learned",
                    bp_iters=16, schedule="PFFPFF", n_apply=32)
    if kind == "train":
        return dict(kind="train", L=rng.randint(6, 12), samples=_log(rng, 200, 2_048), p=p)
    if kind == "bp":
        return dict(kind="bp", L=rng.randint(4, 18), samples=_log(rng, 100, 1_500), p=p, bp_iters=rng.choice([6, 12]),
                    meta=rng.choice([True, False]))
    if kind == "tanner":
        return dict(kind="tanner", classical=rng.choice([40, 80, 120, 200]), samples=_log(rng, 100, 2_000),
                    p=round(rng.uniform(0.005, 0.02), 4), bp_iters=rng.choice([10, 20]), schedule="PFFPFF",
                    n_apply=rng.randint(1, 12))
    return dict(kind="bits", L=rng.randint(4, 16), samples=_log(rng, 200, 20_000), p=round(rng.uniform(0.003, 0.015), 4),
                sweeps=rng.choice([8, 32]))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _bernoulli(shape, p, g):
    """uint8 0/1 array, drawn a slice of rows at a time."""
    out = torch.empty(shape, dtype=torch.uint8, device=DEV)
    step = max(1, (1 << 27) // int(np.prod(shape[1:])))
    for i in range(0, shape[0], step):
        part = out[i:i + step]
        part.copy_(torch.rand(part.shape, device=DEV, generator=g) < p)
    return out


def _words(bits):
    """0/1 bits [n, samples] -> bit-sliced words int64 [n, ceil(samples / 64)]."""
    n, S = bits.shape
    W = (S + 63) // 64
    out = torch.zeros((n, W), dtype=torch.int64, device=bits.device)
    for j in range(64):
        col = bits[:, j::64].to(torch.int64) << j
        out[:, :col.shape[1]] |= col
    return out


_AXIS = {0: -1, 1: -2, 2: -3}     # lattice axis -> dimension of a [..., z, y, x] array


def _plane(n):
    return (1 if n == 0 else 0), (1 if n == 2 else 2)


def _next(t, axis, k=1):
    """t at r + k e_axis."""
    return torch.roll(t, -k, _AXIS[axis])


def _lattice_syndrome(e):
    """Parity of the four edges of every face; e is [..., 3, z, y, x]."""
    out = []
    for n in range(3):
        a, b = _plane(n)
        ea, eb = e[..., a, :, :, :], e[..., b, :, :, :]
        out.append(ea ^ _next(ea, b) ^ eb ^ _next(eb, a))
    return torch.stack(out, -4)


def _measured(c, seed):
    """Errors and one noisy measurement of them as bits [samples, 3, z, y, x]."""
    g = _gen(seed)
    L, S = c["L"], c["samples"]
    e = _bernoulli((S, 3, L, L, L), c["p"], g)
    return e, _lattice_syndrome(e) ^ _bernoulli((S, 3, L, L, L), c["p"], g)


def _slice(bits):
    """[samples, 3, z, y, x] -> bit-sliced words."""
    return _words(bits.reshape(bits.shape[0], -1).T)


def _empty(nbytes):
    return torch.empty(int(nbytes), dtype=torch.uint8, device=DEV)


def _zeros(L, samples):
    return torch.zeros((t3d.n_bits(L), t3d.words_for(samples)), dtype=torch.int64, device=DEV)


@functools.lru_cache(maxsize=None)
def _pretrained():
    """The weights that come with the package (FP32, the order toric3d_cnn_prepare takes)."""
    path = os.path.join(os.path.dirname(t3d.__file__), "weights", "cnn_L12_p04.npz")
    from paper_2212_06985_gb300 import learned
    return learned.load_params(path)


def _gallager(n, rng):
    """Rows of a random classical code with n bits: three permuted partitions into fours
    (column weight 3, row weight 4)."""
    return np.concatenate([rng.permutation(n).reshape(-1, 4) for _ in range(3)])


@functools.lru_cache(maxsize=None)
def _hgp(n):
    """Z checks [m, 7] of the hypergraph product of two such codes, and its qubit count."""
    rng = np.random.default_rng(n)
    r1, r2 = _gallager(n, rng), _gallager(n, rng)
    m = len(r1)
    of_bit = np.argsort(r1.reshape(-1), kind="stable").reshape(n, 3) // 4
    a, j = np.meshgrid(np.arange(n), np.arange(m), indexing="ij")
    bits = a[..., None] * n + r2[j]
    pairs = n * n + of_bit[a] * m + j[..., None]
    checks = np.sort(np.concatenate([bits, pairs], -1).reshape(n * m, 7), axis=1)
    return checks.astype(np.int32), n * n + m * m


def _seed64(seed):
    return int(seed) & 0xFFFFFFFF


# ------------------------------------------------------------------ what a program keeps
def prepare(case, seed):
    c = case
    st = dict(case=c, seed=_seed64(seed), cycle=0)
    kind, S = c["kind"], c.get("samples")
    if kind in ("run", "graph"):
        L = c["L"]
        st["cfg"] = t3d.make_run_cfg(L, c["T"], c["p"], c["p"], st["seed"], S, use_bp=kind == "graph",
                                     bp_iters=c.get("bp_iters", 0), schedule=c["schedule"], n_apply=c["n_apply"],
                                     perfect_round=bool(c.get("perfect", 0)), perfect_max_sweeps=c.get("perfect", 0),
                                     use_graph=kind == "graph")
        st["e"] = _zeros(L, S)
        st["mask"] = torch.zeros(S, dtype=torch.uint8, device=DEV)
        st["counts"] = torch.zeros(8, dtype=torch.int64, device=DEV)
        st["work"] = _empty(t3d.toric3d_run_workspace_bytes(st["cfg"]))
        if kind == "graph":
            st["stream"] = torch.cuda.Stream()
    elif kind == "steps":
        L = c["L"]
        st["e"], st["s"] = _zeros(L, S), _zeros(L, S)
        st["mask"] = torch.zeros(S, dtype=torch.uint8, device=DEV)
        st["counts"] = torch.zeros(8, dtype=torch.int64, device=DEV)
        st["work"] = _empty(t3d.toric3d_flip_workspace_bytes(L, t3d.words_for(S)))
    elif kind == "batch":
        sizes = [c["L"]] + ([c["L2"]] if c["L2"] else [])
        blob = None
        if c["decoder"] == "learned":
            blob = _empty(t3d.toric3d_cnn_blob_bytes())
            t3d.toric3d_cnn_prepare(torch.from_numpy(_pretrained()).to(DEV), blob)
            st["blob"] = blob
        items, st["e"], st["mask"], st["counts"], st["s_prev"], st["fallback"] = [], [], [], [], [], []
        for L in sizes:
            it = dict(L=L, n_samples=S, e=_zeros(L, S), mask=torch.zeros(S, dtype=torch.uint8, device=DEV),
                      counts8=torch.zeros(8, dtype=torch.int64, device=DEV))
            st["e"].append(it["e"])
            st["mask"].append(it["mask"])
            st["counts"].append(it["counts8"])
            if blob is not None:
                it["s_prev"] = _zeros(L, S)
                it["fallback_words"] = torch.zeros(1, dtype=torch.int64, device=DEV)
                st["s_prev"].append(it["s_prev"])
                st["fallback"].append(it["fallback_words"])
            items.append(it)
        st["cfg"] = t3d.make_run_cfg(
            0, 1, c["p"], c["p"], st["seed"], 0, use_bp=c["decoder"] == "bp", bp_iters=c["bp_iters"],
            schedule=c["schedule"], n_apply=c["n_apply"], cnn_blob=blob,
            bp_chunk_samples=16_384 if blob is not None else 0,
            fallback_max_weight=0 if blob is not None else -1, fallback_sigmas=4.0 if blob is not None else 0.0)
        st["batch"] = t3d.make_batch(items)
        st["work"] = _empty(t3d.toric3d_run_batch_workspace_bytes(st["cfg"], st["batch"]))
    elif kind == "bp":
        L = c["L"]
        e, s = _measured(c, seed)
        st["e0"], st["s0"] = _slice(e), _slice(s)
        st["e"], st["s"] = torch.empty_like(st["e0"]), torch.empty_like(st["s0"])
        size = t3d.toric3d_bp_meta_workspace_bytes if c["meta"] else t3d.toric3d_bp_workspace_bytes
        st["work"] = _empty(size(L, S))
        st["llr"] = torch.empty(((2 if c["meta"] else 1), t3d.n_bits(L), S), dtype=torch.float32, device=DEV)
    elif kind == "tanner":
        checks, n = _hgp(c["classical"])
        st["g"] = t3d.tanner_prepare(np.arange(len(checks) + 1, dtype=np.int32) * 7, checks.reshape(-1), n, device=DEV)
        W = t3d.words_for(S)
        st["e0"] = _words(_bernoulli((n, S), c["p"], _gen(seed)))
        st["e"] = torch.empty_like(st["e0"])
        st["s"] = torch.zeros((len(checks), W), dtype=torch.int64, device=DEV)
        st["prior"] = torch.full((n,), math.log((1 - c["p"]) / c["p"]), dtype=torch.float32, device=DEV)
        st["llr"] = torch.empty((n, S), dtype=torch.float32, device=DEV)
        st["work"] = _empty(t3d.toric3d_tanner_bp_workspace_bytes(st["g"], S))
        st["fwork"] = _empty(t3d.toric3d_tanner_flip_workspace_bytes(st["g"], S))
    elif kind == "train":
        L = c["L"]
        sp, s, e = _train_bits(c, seed)
        st["sp"], st["s"], st["label"] = _slice(sp), _slice(s), _slice(e)
        P = torch.from_numpy(_pretrained()).to(DEV)
        st["params"], st["m"] = P.clone(), torch.zeros_like(P)
        st["v"] = torch.full_like(P, 1e-5)      # a run under way: 1,000 steps behind it
        st["step"] = 1_000
        st["blob"] = _empty(t3d.toric3d_cnn_blob_bytes())
        t3d.toric3d_cnn_prepare(st["params"], st["blob"])
        st["loss"] = torch.zeros(1, dtype=torch.float32, device=DEV)
        st["grads"] = torch.zeros_like(P)
        st["work"] = _empty(t3d.toric3d_cnn_train_workspace_bytes(L, S))
    else:
        L = c["L"]
        n, W = t3d.n_bits(L), t3d.words_for(S)
        e = _bernoulli((S, 3, L, L, L), c["p"], _gen(seed))
        st["bits"] = _lattice_syndrome(e).reshape(S, n).contiguous()
        st["e"], st["s"] = _zeros(L, S), _zeros(L, S)
        st["done"] = torch.zeros(1, dtype=torch.int32, device=DEV)
        st["work"] = _empty(t3d.toric3d_flip_until_clear_workspace_bytes(L, W))
        st["fix"] = torch.empty((S, n), dtype=torch.uint8, device=DEV)
        st["left"] = torch.empty((S, n), dtype=torch.uint8, device=DEV)
    return st


def _train_bits(c, seed):
    """Two successive measurements around fresh noise and the error to learn, as bits."""
    g = _gen(seed)
    L, S, p = c["L"], c["samples"], c["p"]
    shape = (S, 3, L, L, L)
    left = _bernoulli(shape, 0.02, g)                     # what the last cycle left behind
    sp = _lattice_syndrome(left) ^ _bernoulli(shape, p, g)
    e = left ^ _bernoulli(shape, p, g)
    return sp, _lattice_syndrome(e) ^ _bernoulli(shape, p, g), e


# ------------------------------------------------------------------ one pass
def run(st):
    c = st["case"]
    kind, S = c["kind"], c.get("samples")
    if kind == "run":                     # a fresh code, then the whole run
        st["e"].zero_()
        t3d.toric3d_run_cycles(st["cfg"], st["e"], st["work"], st["mask"], st["counts"])
        return st["e"], st["mask"], st["counts"]
    if kind == "graph":
        with torch.cuda.stream(st["stream"]):
            st["stream"].wait_stream(torch.cuda.default_stream())
            st["e"].zero_()
            t3d.toric3d_run_cycles(st["cfg"], st["e"], st["work"], st["mask"], st["counts"])
            torch.cuda.default_stream().wait_stream(st["stream"])
        return st["e"], st["mask"], st["counts"]
    if kind == "steps":                   # one cycle of the code in hand, call by call
        st["cycle"] += 1
        L, e, s, t = c["L"], st["e"], st["s"], st["cycle"]
        t3d.toric3d_noise(L, e, c["p"], st["seed"], 0, t)
        t3d.toric3d_syndrome(L, e, s, c["p"], st["seed"], 0, t)
        t3d.toric3d_pflip(L, e, s, c["schedule"], c["n_apply"], 0, st["seed"], 0, t, st["work"])
        t3d.toric3d_logical(L, S, e, st["mask"], st["counts"])
        return e, s, st["mask"], st["counts"]
    if kind == "batch":                   # the next cycle of the codes in hand
        t3d.toric3d_run_batch(st["cfg"], st["batch"], st["work"])
        st["cfg"].cycle0 += 1
        return {k: st[k] for k in ("e", "mask", "counts", "s_prev", "fallback")}
    if kind == "bp":
        st["e"].copy_(st["e0"])
        st["s"].copy_(st["s0"])
        call = t3d.toric3d_bp_meta if c["meta"] else t3d.toric3d_bp
        call(c["L"], S, st["e"], st["s"], c["p"], c["p"], c["bp_iters"], st["work"], st["llr"])
        return st["e"], st["s"], st["llr"]
    if kind == "tanner":
        st["e"].copy_(st["e0"])
        g, e, s = st["g"], st["e"], st["s"]
        t3d.toric3d_tanner_syndrome(g, S, e, s, 0.0, st["seed"], 0, 1)
        t3d.toric3d_tanner_bp(g, S, e, s, st["prior"], c["bp_iters"], st["work"], st["llr"])
        t3d.toric3d_tanner_pflip(g, S, e, s, c["schedule"], c["n_apply"], 0, st["seed"], 0, 1, st["fwork"])
        return e, s, st["llr"]
    if kind == "train":
        st["step"] += 1
        t3d.toric3d_cnn_train_step(c["L"], S, st["sp"], st["s"], st["label"], st["params"], st["m"], st["v"],
                                   st["step"], 1e-3, st["blob"], st["work"], st["loss"], st["grads"])
        return {k: st[k] for k in ("loss", "grads", "params", "m", "v")}
    L, W = c["L"], t3d.words_for(S)
    n = t3d.n_bits(L)
    t3d.toric3d_pack(n, S, st["bits"], st["s"])
    st["e"].zero_()
    t3d.toric3d_flip_until_clear(L, st["e"], st["s"], c["sweeps"], st["work"], st["done"])
    t3d.toric3d_unpack(n, S, st["e"], st["fix"])
    t3d.toric3d_unpack(n, S, st["s"], st["left"])
    return st["fix"], st["left"], st["done"]


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    c = case
    kind, S = c["kind"], c.get("samples")
    if kind == "tanner":
        checks, n = _hgp(c["classical"])
        W, m, E = t3d.words_for(S), len(checks), checks.size
        # e in, e and s out, posteriors out; a message update: 3 adds, a tanh and an atanh (4
        # operations each), two products and a sign / clamp
        return dict(bytes=8.0 * W * (2 * n + m) + 4.0 * n * S, flops=16.0 * E * S * c["bp_iters"])
    L = c["L"]
    n, W = 3 * L ** 3, (S + 63) // 64
    if kind == "run" or kind == "graph":
        # a fresh code needs no input; the state and the readout come out
        return dict(bytes=8.0 * n * W + S + 64, flops=64.0 * n * S * c.get("bp_iters", 0) * c["T"])
    if kind == "steps":
        return dict(bytes=8.0 * W * n * 3 + S + 64, flops=0.0)
    if kind == "batch":
        n2 = 3 * c["L2"] ** 3
        k = 2 if c["L2"] else 1
        state = 2 * 8.0 * (n + n2) * W + k * (S + 64)
        if c["decoder"] == "learned":
            # s_prev in and out as well; the three convolutions and the head
            return dict(bytes=state + 2 * 8.0 * n * W, flops=32_928.0 * L ** 3 * S)
        return dict(bytes=state, flops=64.0 * (n + n2) * S * c["bp_iters"])
    if kind == "bp":
        meta = c["meta"]
        # with meta-checks: a fifth message per face and six per cube (two per face)
        return dict(bytes=4 * 8.0 * n * W + 4.0 * n * S * (2 if meta else 1),
                    flops=(112.0 if meta else 64.0) * n * S * c["bp_iters"])
    if kind == "train":
        # three bit arrays in; forward, backward data (two layers) and weight gradients
        macs = 27 * 16 * (6 + 16 + 16) + 48
        back = 27 * 16 * (16 + 16) + 48
        return dict(bytes=3 * 8.0 * n * W + 16_515 * 4.0 * 7, flops=2.0 * L ** 3 * S * (2 * macs + back))
    return dict(bytes=3.0 * n * S, flops=0.0)


# ------------------------------------------------------------------ the same numbers in 64 bits
def _check64(x, sign, extra=1.0):
    """Outgoing messages of a check over the inputs x (last dimension), one by one."""
    t = torch.tanh(x / 2)
    k = x.shape[-1]
    out = []
    for i in range(k):
        prod = torch.full_like(t[..., 0], extra)
        for j in range(k):
            if j != i:
                prod = prod * t[..., j]
        out.append((2 * torch.atanh(prod.clamp(-1 + 1e-15, 1 - 1e-15))).clamp(-30, 30) * sign)
    return out


def _lattice_bp64(s, p, iters, meta):
    """Posteriors [2 or 1, 3, z, y, x] of flooding BP per sample, FP64; s is [samples, 3, z, y, x]."""
    sg = 1.0 - 2.0 * s.double()
    l0 = math.log((1 - p) / p)
    shape = s[:, 0].shape
    zero = torch.zeros(shape, dtype=torch.float64, device=s.device)
    M = [[zero] * 4 for _ in range(3)]
    up, lo, hi = [zero] * 3, [zero] * 3, [zero] * 3       # face, lower cube and upper cube -> measurement variable

    def totals():
        T = [zero + l0 for _ in range(3)]
        for n in range(3):
            a, b = _plane(n)
            T[a] = T[a] + M[n][0] + _next(M[n][1], b, -1)
            T[b] = T[b] + M[n][2] + _next(M[n][3], a, -1)
        return T

    for _ in range(iters):
        T = totals()
        new = []
        for n in range(3):
            a, b = _plane(n)
            x = [T[a] - M[n][0], _next(T[a], b) - M[n][1], T[b] - M[n][2], _next(T[b], a) - M[n][3]]
            if meta:
                x.append(l0 + lo[n] + hi[n])
            new.append(_check64(torch.stack(x, -1), sg[:, n], 1.0 if meta else math.tanh(l0 / 2)))
        if meta:
            x, par = [], 1.0
            for n in range(3):
                x += [l0 + up[n] + hi[n], _next(l0 + up[n] + lo[n], n)]
                par = par * sg[:, n] * _next(sg[:, n], n)
            c = _check64(torch.stack(x, -1), par)
            lo = [c[2 * n] for n in range(3)]
            hi = [_next(c[2 * n + 1], n, -1) for n in range(3)]
            up = [new[n][4] for n in range(3)]
        M = [m[:4] for m in new]
    T = torch.stack(totals(), 1)
    if not meta:
        return T[None]
    return torch.stack([T, torch.stack([l0 + up[n] + lo[n] + hi[n] for n in range(3)], 1)])


def _exact_bp(c, seed):
    _, s = _measured(c, seed)
    S, n = c["samples"], 3 * c["L"] ** 3
    out = torch.empty(((2 if c["meta"] else 1), n, S), dtype=torch.float64, device=DEV)
    step = max(1, (1 << 22) // n)
    for i in range(0, S, step):
        l = _lattice_bp64(s[i:i + step], c["p"], c["bp_iters"], c["meta"])
        out[:, :, i:i + step] = l.reshape(l.shape[0], l.shape[1], n).transpose(1, 2)
    return None, None, out


def _exact_tanner(c, seed):
    checks, n = _hgp(c["classical"])
    C = torch.from_numpy(checks.astype(np.int64)).to(DEV)
    S = c["samples"]
    e = _bernoulli((n, S), c["p"], _gen(seed))
    out = torch.empty((n, S), dtype=torch.float64, device=DEV)
    l0 = math.log((1 - c["p"]) / c["p"])
    step = max(1, (1 << 25) // checks.size)
    for i in range(0, S, step):
        b = e[:, i:i + step]
        syn = b[C[:, 0]].clone()
        for k in range(1, 7):
            syn ^= b[C[:, k]]
        sg = 1.0 - 2.0 * syn.double()
        M = torch.zeros((len(checks), 7, b.shape[1]), dtype=torch.float64, device=DEV)
        for it in range(c["bp_iters"] + 1):
            T = torch.full((n, b.shape[1]), l0, dtype=torch.float64, device=DEV)
            T.index_add_(0, C.reshape(-1), M.reshape(-1, b.shape[1]))
            if it < c["bp_iters"]:
                M = torch.stack(_check64((T[C.reshape(-1)].reshape(M.shape) - M).transpose(1, 2), sg), 1)
        out[:, i:i + step] = T
    return None, None, out


_SHAPES = [(16, 6, 3, 3, 3), (16,), (16, 16, 3, 3, 3), (16,), (16, 16, 3, 3, 3), (16,), (3, 16), (3,)]


def _exact_train(c, seed):
    import torch.nn.functional as F
    sp, s, e = _train_bits(c, seed)
    L, S = c["L"], c["samples"]
    P = torch.from_numpy(_pretrained()).to(DEV)
    parts, i = [], 0
    for sh in _SHAPES:
        k = int(np.prod(sh))
        parts.append(P[i:i + k].double().reshape(sh).requires_grad_())
        i += k
    total = 0.0
    for k in range(0, S, 128):
        h = torch.cat([sp[k:k + 128], s[k:k + 128]], 1).double()
        for layer in range(3):
            h = F.pad(h, (1,) * 6, mode="circular")
            h = torch.relu(F.conv3d(h, parts[2 * layer], parts[2 * layer + 1]))
        z = torch.einsum("scabd,ec->seabd", h, parts[6]) + parts[7].view(1, -1, 1, 1, 1)
        loss = F.binary_cross_entropy_with_logits(z, e[k:k + 128].double(), reduction="sum")
        (loss / (3 * L ** 3 * S)).backward()
        total += float(loss.detach())
    g = torch.cat([q.grad.reshape(-1) for q in parts])
    m, v = 0.1 * g, 0.999 * 1e-5 + 0.001 * g * g
    c1, c2 = 1 - 0.9 ** 1_001, 1 - 0.999 ** 1_001
    params = P.double() - 1e-3 * (m / c1) / (torch.sqrt(v / c2) + 1e-8)
    loss = torch.tensor([total], dtype=torch.float64, device=DEV)
    return dict(loss=loss, grads=g, params=params, m=m, v=v)


def exact(case, seed):
    c = case
    if c["kind"] == "bp":
        return _exact_bp(c, seed)
    if c["kind"] == "tanner":
        return _exact_tanner(c, seed)
    if c["kind"] == "train":
        return _exact_train(c, seed)
    return None       # error states, masks and counts: whole numbers
