"""Faster routes of the BP decoders against the plain ones, bit for bit.  The first two iterations in one launch
(toric3d_bp) against the same iterations one by one (toric3d_bp_step): posteriors for one to four iterations,
with and without measurement-error variables, on lattices where every neighbour wraps (L = 2, 3) and larger
ones, ragged batches, chunked and whole; the meta-check decode and the low-degree Tanner iteration likewise."""
import numpy as np
import pytest
import torch

import paper_2212_06985_gb300 as t3d
import toric3d_inputs as inp
from gpu_util import dev, upload_bits, workspace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q", [0.0, 0.04])
@pytest.mark.parametrize("L,S", [(2, 70), (3, 64), (5, 130), (8, 1)])
@pytest.mark.parametrize("iters", [1, 2, 3, 4])
def test_decode_equals_single_iterations(L, S, iters, q):
    n = 3 * L ** 3
    s = upload_bits(inp.random_bits(S, n, 0.2, seed=L + S))
    e = torch.zeros_like(s)
    msg = [torch.empty(t3d.toric3d_bp_message_bytes(L, S) // 4, dtype=torch.float32, device=dev()) for _ in range(2)]
    for k in range(iters):
        t3d.toric3d_bp_step(L, S, s, 0.04, q, msg[(k + 1) % 2] if k else None, msg[k % 2])
    want = torch.empty((n, S), dtype=torch.float32, device=dev())
    we, ws = e.clone(), s.clone()
    t3d.toric3d_bp_decide(L, S, msg[(iters - 1) % 2], 0.04, we, ws,
                          workspace(t3d.toric3d_bp_decide_workspace_bytes(L, S)), want)
    got = torch.empty_like(want)
    ge, gs = e.clone(), s.clone()
    t3d.toric3d_bp(L, S, ge, gs, 0.04, q, iters, workspace(t3d.toric3d_bp_workspace_bytes(L, S)), got)
    assert torch.equal(got, want) and torch.equal(ge, we) and torch.equal(gs, ws)
    ge, gs = e.clone(), s.clone()
    t3d.toric3d_bp(L, S, ge, gs, 0.04, q, iters, workspace(t3d.toric3d_bp_workspace_bytes(L, 64)))
    assert torch.equal(ge, we) and torch.equal(gs, ws)


@pytest.mark.parametrize("L,S", [(2, 70), (3, 64), (4, 300), (6, 1)])
@pytest.mark.parametrize("iters", [0, 1, 2, 3])
def test_meta_decode_equals_single_iterations(L, S, iters):
    """The meta-check decode (whose first iteration reads no messages) against toric3d_bp_meta_step from
    an all-zero buffer: every posterior is the prior plus that step's messages, summed in their order."""
    n, n3 = 3 * L ** 3, L ** 3
    s = upload_bits(inp.random_bits(S, n, 0.2, seed=L + S))
    Sp = 64 * inp.words_for(S)
    msg = [torch.zeros((7 * n, Sp), dtype=torch.float32, device=dev()) for _ in range(2)]
    work = workspace(n * Sp * 4)
    for k in range(iters):
        t3d.toric3d_bp_meta_step(L, S, s, 0.04, 0.03, msg[k % 2], msg[(k + 1) % 2], work)
    m = msg[iters % 2]
    F = m[:4 * n].view(3, L, L, L, 4, Sp)
    l0 = torch.log(torch.tensor((1 - 0.04) / 0.04, dtype=torch.float64)).float().item()
    lq = torch.log(torch.tensor((1 - 0.03) / 0.03, dtype=torch.float64)).float().item()
    axis = {0: 2, 1: 1, 2: 0}                        # lattice axis -> dimension of a [z, y, x, ...] array
    want = torch.empty((2, n, Sp), dtype=torch.float32, device=dev())
    for d in range(3):
        t = torch.full((L, L, L, Sp), l0, dtype=torch.float32, device=dev())
        for nn in [k for k in range(3) if k != d]:
            ax = 3 - d - nn
            lo = 0 if d < ax else 2
            t = t + F[nn, :, :, :, lo]
            t = t + torch.roll(F[nn, :, :, :, lo + 1], 1, axis[ax])
        want[0, d * n3:(d + 1) * n3] = t.reshape(n3, Sp)
    want[1] = ((lq + m[4 * n:5 * n]) + m[5 * n:6 * n]) + m[6 * n:7 * n]
    got = torch.empty((2, n, S), dtype=torch.float32, device=dev())
    e = torch.zeros_like(s)
    t3d.toric3d_bp_meta(L, S, e, s.clone(), 0.04, 0.03, iters, workspace(t3d.toric3d_bp_meta_workspace_bytes(L, S)), got)
    assert torch.equal(got, want[:, :, :S])
    bits = (want[0] < 0)[:, :S].cpu().numpy().astype("uint8")
    assert (e.cpu().numpy().view("uint64") == inp.pack(bits.T)).all()


def _low_degree_code(n, m, seed):
    """Checks of degree 0 .. 8, every variable in at most four; one variable in none."""
    rng = np.random.default_rng(seed)
    room = np.full(n, 4)
    room[n // 2] = 0
    rows = []
    for c in range(m):
        free = np.nonzero(room)[0]
        row = rng.choice(free, min(len(free), c % 9), replace=False)
        room[row] -= 1
        rows.append(sorted(int(v) for v in row))
    return rows


@pytest.mark.parametrize("S,iters", [(64, 0), (1, 1), (70, 2), (130, 3), (300, 7)])
@pytest.mark.parametrize("seed", [1, 2])
def test_low_degree_graphs_equal_the_general_kernels(S, iters, seed):
    """The one-kernel Tanner iteration against the general two kernels: the same code with a check of
    degree nine on nine further variables appended takes the general ones; messages, posteriors and
    corrections of the shared part equal bit for bit."""
    n, m = 60, 40
    rows = _low_degree_code(n, m, seed)
    graphs = []
    for extra in (False, True):
        r = rows + ([list(range(n, n + 9))] if extra else [])
        cptr = np.concatenate([[0], np.cumsum([len(x) for x in r])]).astype(np.int32)
        cvar = np.array([v for x in r for v in x], dtype=np.int32)
        graphs.append(t3d.tanner_prepare(cptr, cvar, n + (9 if extra else 0)))
    assert graphs[0].desc.max_check_degree == 8 and graphs[1].desc.max_check_degree == 9
    assert graphs[0].desc.max_var_degree <= 4
    rng = np.random.default_rng(seed + S)
    ebits = (rng.random((S, n + 9)) < 0.1).astype(np.uint8)
    sbits = (rng.random((S, m + 1)) < 0.3).astype(np.uint8)
    prior = torch.from_numpy(rng.normal(2.0, 1.5, n + 9).astype(np.float32)).to(dev())
    out = []
    for g in graphs:
        k = g.n_vars
        e, s = upload_bits(ebits[:, :k]), upload_bits(sbits[:, :g.n_checks])
        llr = torch.empty((k, S), dtype=torch.float32, device=dev())
        t3d.toric3d_tanner_bp(g, S, e, s, prior[:k].contiguous(), iters,
                              workspace(t3d.toric3d_tanner_bp_workspace_bytes(g, S)), llr)
        Sp = 64 * inp.words_for(S)
        msg = [torch.zeros((g.n_edges, Sp), dtype=torch.float32, device=dev()) for _ in range(2)]
        syn = upload_bits(sbits[:, :g.n_checks])
        for i in range(iters):
            t3d.toric3d_tanner_bp_step(g, S, syn, prior[:k].contiguous(), msg[i % 2], msg[(i + 1) % 2],
                                       workspace(k * Sp * 4))
        out.append((llr[:n], e[:n], s[:m], msg[iters % 2][:graphs[0].n_edges]))
    for a, b in zip(*out):
        assert torch.equal(a, b)
