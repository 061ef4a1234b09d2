"""The measurement on both sides of the line between a face a thread (fewer than 240 blocks of sites) and sites a
thread: one word to several word tiles, the last one partial, noiseless, noisy and always flipped, and a
batch whose items together cross the line, against the oracle bit for bit."""
import numpy as np
import pytest
import torch

import oracle
import paper_2212_06985_gb300 as t3d
import toric3d_inputs as inp
from gpu_util import dev, download_bits, workspace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,W", [(2, 1), (3, 5), (12, 32), (12, 33), (9, 64), (9, 65), (5, 470), (5, 520), (20, 4), (20, 9)])
@pytest.mark.parametrize("q", [0.0, 0.03, 1.0])
def test_measurement_matches_oracle(L, W, q):
    n = 3 * L ** 3
    e = torch.zeros((n, W), dtype=torch.int64, device=dev())
    s = torch.full_like(e, 5)
    t3d.toric3d_noise(L, e, 0.1, 7, 192, 3)
    t3d.toric3d_syndrome(L, e, s, q, 8, 192, 3)
    for w in {0, W // 2, W - 1}:
        ew = download_bits(e[:, w:w + 1].contiguous(), 64)
        want = oracle.measure_batch(L, ew, q, 8, 192 + 64 * w, 3)
        assert np.array_equal(download_bits(s[:, w:w + 1].contiguous(), 64), want), w


@pytest.mark.parametrize("specs", [[(4, 100), (6, 700)], [(9, 2100), (10, 2100), (3, 65)]])
def test_batch_matches_single_runs(specs):
    T, kw = 2, dict(schedule="PF", n_apply=2)
    items = [dict(L=L, n_samples=S, sample0=64000 * i, e=torch.zeros((3 * L ** 3, inp.words_for(S)), dtype=torch.int64,
                                                                      device=dev())) for i, (L, S) in enumerate(specs)]
    batch = t3d.make_batch(items)
    cfg = t3d.make_run_cfg(4, T, 0.04, 0.04, 3, 1, **kw)
    t3d.toric3d_run_batch(cfg, batch, workspace(t3d.toric3d_run_batch_workspace_bytes(cfg, batch)))
    for item, (L, S) in zip(items, specs):
        k = min(S, 70)
        _, want = oracle.run_batch(oracle.make_cfg(L, T, 0.04, 0.04, 3, **kw), item["sample0"], k)
        assert np.array_equal(download_bits(item["e"], S)[:k], want), L
