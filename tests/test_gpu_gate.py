"""The fallback gate's counters against CPU weights: fewer faces than a thread's seven, one and many
face ranges, counts at the top of a counter's bits (all faces unsatisfied), ragged word tiles."""
import numpy as np
import pytest
import torch

import paper_2212_06985_gb300 as t3d
from gpu_util import dev, upload_bits, workspace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,S", [(2, 70), (3, 64 * 33), (5, 64 * 31 + 1), (12, 700), (20, 130), (13, 64 * 64)])
def test_gate_counts_match_cpu_weights(L, S):
    n = 3 * L ** 3
    rng = np.random.default_rng(L)
    bits = (rng.random((S, n)) < rng.uniform(0.0, 1.0, S)[:, None]).astype(np.uint8)
    bits[S // 2] = 1
    s = upload_bits(bits)
    W = s.shape[1]
    weight = np.zeros(W * 64, dtype=np.int64)
    weight[:S] = bits.sum(axis=1)
    work = workspace(t3d.toric3d_gate_workspace_bytes(L, W))
    tops = np.sort(weight.reshape(W, 64).max(axis=1))
    for max_w in {0, n // 2, int(tops[0]), int(tops[W // 2]), int(tops[W // 2]) - 1, n - 1, n}:
        gate = torch.full((W,), 7, dtype=torch.uint8, device=dev())
        count = torch.zeros(1, dtype=torch.int64, device=dev())
        t3d.toric3d_gate(L, s, max(max_w, 0), gate, work, count)
        want = (weight.reshape(W, 64) > max(max_w, 0)).any(axis=1)
        assert np.array_equal(gate.cpu().numpy().astype(bool), want), max_w
        assert int(count.item()) == int(want.sum())
