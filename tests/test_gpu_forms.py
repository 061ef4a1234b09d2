"""Both forms of a schedule at sizes where the other one is usually taken, against the oracle bit for bit on
the first, a middle and the last word of the batch: the step kernels on lattices that also fit on
chip (flip tiles of 256 threads and, at L = 32, of 1,024; p-flip's two passes; an odd number of flips,
which is copied back), and the on-chip form whose columns are turned (64 words or more, row tiles that are
not a multiple of 32 at odd L).  Launch counts say which form ran."""
import numpy as np
import pytest
import torch

import oracle
import paper_2212_06985_gb300 as t3d
import toric3d_inputs as inp
from gpu_util import dev, download_bits, workspace
from test_gpu_learned import _blob, _run, _stepwise
from test_gpu_routes import count_launches

pytestmark = pytest.mark.gpu

SEED, SAMPLE0, CYCLE, SWEEP0 = 5, 128, 2, 9


def noisy(L, W, p, q):
    e = torch.zeros((3 * L ** 3, W), dtype=torch.int64, device=dev())
    s = torch.zeros_like(e)
    t3d.toric3d_noise(L, e, p, SEED, SAMPLE0, CYCLE)
    t3d.toric3d_syndrome(L, e, s, q, SEED, SAMPLE0, CYCLE)
    return e, s


def column(words, w):
    return download_bits(words[:, w:w + 1].contiguous(), 64)


def check_schedule(L, W, schedule, n, run, p=0.03):
    """run(e, s, work) in place; returns its flip and p-flip launches."""
    e, s = noisy(L, W, p, p)
    checked = sorted({0, W // 2, W - 1})
    before = {w: (column(e, w), column(s, w)) for w in checked}
    work = workspace(t3d.toric3d_flip_workspace_bytes(L, W))
    launches = count_launches(lambda: run(e, s, work), "flip", "pflip")
    for w in checked:
        we, ws = before[w]
        for k in range(n):
            we, ws = oracle.flip_batch(L, we, ws, probabilistic=schedule[k % len(schedule)] == "P", seed=SEED,
                                       sample0=SAMPLE0 + 64 * w, cycle=CYCLE, sweep=SWEEP0 + k)
        assert np.array_equal(column(e, w), we) and np.array_equal(column(s, w), ws), w
    return launches


def pflip(L, schedule, n):
    return lambda e, s, work: t3d.toric3d_pflip(L, e, s, schedule, n, SWEEP0, SEED, SAMPLE0, CYCLE, work)


# sizes where the estimate for the other form is at least a fifth higher
@pytest.mark.parametrize("L,W,schedule,n", [(12, 2000, "F", 2), (14, 160, "PF", 2), (16, 65, "P", 2), (16, 701, "F", 2),
                                            (18, 331, "FFP", 3), (25, 200, "FPFP", 4), (24, 301, "FFP", 3),
                                            (24, 70, "P", 2), (26, 313, "FFPFF", 5), (31, 65, "FP", 2),
                                            (31, 97, "PFF", 3), (32, 330, "F", 2), (32, 161, "F", 1), (32, 16, "P", 2)])
def test_step_kernels_match_oracle(L, W, schedule, n):
    letters = (schedule * n)[:n]
    assert check_schedule(L, W, schedule, n, pflip(L, schedule, n)) == [letters.count("F"), letters.count("P")]


@pytest.mark.parametrize("L,W", [(15, 64), (16, 69), (17, 66), (21, 70), (23, 66), (31, 66), (32, 65)])
def test_turned_columns_match_oracle(L, W):
    # one launch to turn the columns, the schedule, two turning back under one count
    schedule = "FFFPFFF"
    assert sum(check_schedule(L, W, schedule, 7, pflip(L, schedule, 7))) == 3


@pytest.mark.parametrize("L,W", [(15, 64), (17, 66), (23, 67), (26, 66), (31, 66)])   # clusters of 1, 2, 4, 7, 8
@pytest.mark.parametrize("p,most", [(0.002, 40), (0.05, 11)])   # clears early (L = 31 keeps a stuck pair); does not
def test_until_clear_with_turned_columns_matches_oracle(L, W, p, most):
    e, s = noisy(L, W, p, 0.0)
    used = [0, W // 2, W - 1]   # errors in these words alone, so that the oracle sees every application
    keep = torch.zeros(W, dtype=torch.int64, device=dev())
    keep[used] = -1
    e &= keep
    s &= keep
    want = []
    for w in used:
        want.append([column(e, w), column(s, w)])
    count = 0
    while count < most and any(ws.any() for _, ws in want):
        want = [oracle.flip_batch(L, we, ws) for we, ws in want]
        count += 1
    done = torch.full((1,), -5, dtype=torch.int32, device=dev())
    work = workspace(t3d.toric3d_flip_until_clear_workspace_bytes(L, W))
    launches = count_launches(lambda: t3d.toric3d_flip_until_clear(L, e, s, most, work, done), "flip")
    assert launches == [3]
    assert int(done.item()) == count
    for w, (we, ws) in zip(used, want):
        assert np.array_equal(column(e, w), we) and np.array_equal(column(s, w), ws), w
    e &= ~keep
    s &= ~keep
    assert not e.any() and not s.any()


@pytest.mark.parametrize("L,W,most", [(16, 160, 1), (28, 70, 3), (32, 160, 1)])
def test_until_clear_step_by_step_matches_oracle(L, W, most):
    e, s = noisy(L, W, 0.03, 0.0)
    used = [0, W - 1]
    want = [[column(e, w), column(s, w)] for w in used]
    for _ in range(most):
        want = [oracle.flip_batch(L, we, ws) for we, ws in want]
    done = torch.full((1,), -5, dtype=torch.int32, device=dev())
    work = workspace(t3d.toric3d_flip_until_clear_workspace_bytes(L, W))
    t3d.toric3d_flip_until_clear(L, e, s, most, work, done)
    assert int(done.item()) == most
    for w, (we, ws) in zip(used, want):
        assert np.array_equal(column(e, w), we) and np.array_equal(column(s, w), ws), w


@pytest.mark.parametrize("L,W", [(16, 66), (15, 200), (16, 9), (32, 40)])
def test_flip_without_allocation_matches_oracle(L, W):
    # the schedule's columns are turned in the library's own scratch array
    check_schedule(L, W, "F", 5, lambda e, s, work: t3d.toric3d_flip_noalloc(L, e, s, 5))


def test_batch_of_both_forms_with_a_noiseless_round():
    # L = 8 with 100,000 samples runs whole on chip, the others step by step with the noiseless round
    T, specs = 2, [(8, 100_000, 0), (20, 500, 100_032), (33, 130, 100_608)]
    kw = dict(schedule="FFPFF", n_apply=5, perfect_round=True, perfect_max_sweeps=4)
    items = [dict(L=L, n_samples=S, sample0=o, mask=torch.zeros(S, dtype=torch.uint8, device=dev()),
                  e=torch.zeros((3 * L ** 3, inp.words_for(S)), dtype=torch.int64, device=dev())) for L, S, o in specs]
    batch = t3d.make_batch(items)
    cfg = t3d.make_run_cfg(8, T, 0.03, 0.03, 11, 1, **kw)
    work = workspace(t3d.toric3d_run_batch_workspace_bytes(cfg, batch))
    assert count_launches(lambda: t3d.toric3d_run_batch(cfg, batch, work), "noise", "syndrome") == [T, T + 1]
    for item, (L, S, o) in zip(items, specs):
        W = inp.words_for(S)
        for w in {0, W - 1}:
            k = min(64, S - 64 * w)
            want_mask, want_e = oracle.run_batch(oracle.make_cfg(L, T, 0.03, 0.03, 11, **kw), o + 64 * w, k)
            assert np.array_equal(column(item["e"], w)[:k], want_e), (L, w)
            assert np.array_equal(item["mask"][64 * w:64 * w + k].cpu().numpy(), want_mask), (L, w)


@pytest.mark.parametrize("L,S", [(15, 64 * 66 + 5), (17, 64 * 20)])
def test_learned_fallback_on_some_words_equals_stepwise(L, S):
    # the flagged words' schedule runs on chip over a compacted copy, each word with its own coins
    T, W, blob = 2, inp.words_for(S), _blob(3)
    lo, hi = 0, 3 * L ** 3   # thresholds that flag every word and none
    while hi - lo > 1:
        mid = (lo + hi) // 2
        fb = _run(L, S, T, blob, mid)[2]
        if 0.2 * T * W <= fb <= 0.8 * T * W:
            break
        lo, hi = (mid, hi) if fb > 0.5 * T * W else (lo, mid)
    e_ref, sp_ref, flagged = _stepwise(L, S, T, blob, mid)
    e, sp, fb, counts = _run(L, S, T, blob, mid)
    assert 0 < fb < T * W and fb == flagged
    assert np.array_equal(e, e_ref) and np.array_equal(sp, sp_ref) and counts.sum() == S
