"""Unpacking on both sides of 400,000 bytes (a byte a thread up to there; 1,000,000 in one word) and where the tiles are split over one, two,
four and eight blocks by samples, rows that are and are not 4-byte aligned, a partial last word."""
import numpy as np
import pytest
import torch

import paper_2212_06985_gb300 as t3d
import toric3d_inputs as inp
from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,S", [(1, 1), (5, 63), (400_000, 1), (400_001, 1), (1000, 400), (1000, 401), (999, 400), (999, 402),
                                 (15_625, 64), (15_626, 64), (640, 1100), (2304, 1061), (4999, 1025), (9601, 130), (5184, 577)])
def test_unpack_matches_reference(n, S):
    rng = np.random.default_rng(n + S)
    raw = rng.integers(0, 2, (S, n), dtype=np.uint8)
    words = torch.from_numpy(inp.pack(raw).view(np.int64)).to(dev())
    room = torch.full((S * n + 64,), 0xAA, dtype=torch.uint8, device=dev())
    bits = room[32:32 + S * n].view(S, n)
    t3d.toric3d_unpack(n, S, words, bits)
    assert np.array_equal(bits.cpu().numpy(), raw)
    rest = torch.cat([room[:32], room[32 + S * n:]])
    assert int(rest.min()) == int(rest.max()) == 0xAA
