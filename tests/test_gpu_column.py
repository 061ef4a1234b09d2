"""Lattices kept on one SM or a cluster (t3d_column.cu) against the oracle, bit for bit: the smallest
(several words per block), odd ones, the largest with the error words in shared memory (L = 14) and
beside it (15, 16), every cluster size the larger ones take (17 .. 32, equal and unequal slabs), the
first that goes step by step (33); ragged batches, a starting error,
schedules that do and do not cycle, more than one cycle, sample0, and the noise extremes 0 and 1."""
import numpy as np
import pytest
import torch

import oracle
import paper_2212_06985_gb300 as t3d
import toric3d_inputs as inp
from gpu_util import dev, download_bits, upload_bits, workspace, zeros_words

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,S,T,p,schedule,n_apply,perfect,graph",
                         [(2, 1000, 3, 0.05, "FP", 3, 8, False), (3, 65, 2, 0.04, "PFFPFF", 8, -1, False),
                          (4, 10_000, 2, 0.02, "F", 7, 32, True), (5, 130, 3, 1.0, "P", 2, -1, False),
                          (7, 100, 2, 0.04, "FFPFF", 5, 16, False), (13, 64, 1, 0.03, "FFPFF", 6, -1, False),
                          (14, 70, 2, 0.04, "PF", 4, 4, False), (15, 33, 2, 0.04, "PFF", 4, 4, False),
                          (16, 66, 2, 0.03, "FFPFF", 5, 6, True), (17, 20, 2, 0.04, "FFPFF", 5, 4, False),
                          (6, 64, 0, 0.02, "F", 1, 10, False), (4, 64, 2, 0.0, "F", 0, 3, False)])
def test_runs_match_oracle(L, S, T, p, schedule, n_apply, perfect, graph):
    n, s0 = 3 * L ** 3, 128
    kw = dict(schedule=schedule, n_apply=n_apply, perfect_round=perfect >= 0, perfect_max_sweeps=max(perfect, 0))
    start = inp.random_bits(S, n, 0.03, seed=L)
    cfg = t3d.make_run_cfg(L, T, p, p, 77, S, sample0=s0, cycle0=3, use_graph=graph, **kw)
    e = upload_bits(start)
    work = workspace(t3d.toric3d_run_workspace_bytes(cfg))
    mask = torch.zeros(S, dtype=torch.uint8, device=dev())
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        t3d.toric3d_run_cycles(cfg, e, work, mask)
    torch.cuda.synchronize()
    k = min(S, 200)
    ora_mask, ora_e = oracle.run_batch(oracle.make_cfg(L, T, p, p, 77, cycle0=3, **kw), s0, k, start[:k])
    assert np.array_equal(download_bits(e, S)[:k], ora_e)
    assert np.array_equal(mask.cpu().numpy()[:k], ora_mask)


@pytest.mark.parametrize("L", [2, 3, 4, 9, 14, 15, 16, 17, 20, 23, 26, 27, 30, 31, 32, 33])
@pytest.mark.parametrize("S", [40, 200])
def test_sweeps_and_until_clear_match_oracle(L, S):
    n, W = 3 * L ** 3, inp.words_for(S)
    ebits = inp.random_bits(S, n, 0.01, seed=L)
    sbits = oracle.syndrome_batch(L, ebits)
    e, s = upload_bits(ebits), upload_bits(sbits)
    work = workspace(t3d.toric3d_flip_workspace_bytes(L, W))
    t3d.toric3d_pflip(L, e, s, "FPP", 4, 9, 5, 64, 2, work)
    we, ws = ebits.copy(), sbits.copy()
    for k in range(4):
        we, ws = oracle.flip_batch(L, we, ws, probabilistic="FPP"[k % 3] == "P", seed=5, sample0=64, cycle=2, sweep=9 + k)
    assert np.array_equal(download_bits(e, S), we) and np.array_equal(download_bits(s, S), ws)

    e, s = upload_bits(ebits), upload_bits(sbits)
    work = workspace(t3d.toric3d_flip_until_clear_workspace_bytes(L, W))
    done = torch.full((1,), -5, dtype=torch.int32, device=dev())
    t3d.toric3d_flip_until_clear(L, e, s, 6, work, done)
    we, ws, count = ebits.copy(), sbits.copy(), 0
    while count < 6 and ws.any():
        we, ws = oracle.flip_batch(L, we, ws)
        count += 1
    assert np.array_equal(download_bits(e, S), we) and np.array_equal(download_bits(s, S), ws)
    assert int(done.item()) == count
    clear = zeros_words(n, S)
    t3d.toric3d_flip_until_clear(L, e, clear, 6, work, done)
    assert int(done.item()) == 0 and not clear.any()


@pytest.mark.parametrize("L,S,T,schedule,n_apply", [(3, 129, 3, "F", 0), (6, 64 * 700 + 9, 2, "FP", 3),
                                                    (8, 64 * 400, 2, "FFPFF", 5), (10, 64 * 310 + 5, 2, "PF", 2),
                                                    (11, 64 * 3 + 1, 2, "PF", 2)])
def test_runs_with_a_thread_per_site_match_oracle(L, S, T, schedule, n_apply):
    # L = 10 is the largest lattice with a thread per site, L = 11 the first without; more columns than
    # blocks resident at once; n_apply = 0: measurements follow each other directly
    n = 3 * L ** 3
    kw = dict(schedule=schedule, n_apply=n_apply, perfect_round=True, perfect_max_sweeps=3)
    start = inp.random_bits(S, n, 0.02, seed=L)
    cfg = t3d.make_run_cfg(L, T, 0.03, 0.03, 78, S, sample0=64, cycle0=1, use_graph=False, **kw)
    e, mask = upload_bits(start), torch.zeros(S, dtype=torch.uint8, device=dev())
    t3d.toric3d_run_cycles(cfg, e, workspace(t3d.toric3d_run_workspace_bytes(cfg)), mask)
    got_e, got_mask = download_bits(e, S), mask.cpu().numpy()
    for a in {0, (S - 1) // 64 * 64}:   # the first words and the last
        k = min(S - a, 100)
        want_mask, want_e = oracle.run_batch(oracle.make_cfg(L, T, 0.03, 0.03, 78, cycle0=1, **kw), 64 + a, k,
                                             start[a:a + k])
        assert np.array_equal(got_e[a:a + k], want_e) and np.array_equal(got_mask[a:a + k], want_mask)
