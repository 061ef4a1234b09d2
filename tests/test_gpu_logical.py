"""The logical readout's tiles against the oracle: two, four and eight words (one block per SM at
most), and the serial kernel above; ragged last words and tiles, one line row and several."""
import numpy as np
import pytest
import torch

import oracle
import paper_2212_06985_gb300 as t3d
import toric3d_inputs as inp
from gpu_util import dev, upload_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,S", [(2, 1), (3, 65), (13, 129), (17, 130), (4, 64 * 304), (4, 64 * 304 + 1),
                                 (5, 64 * 608 - 5), (3, 64 * 608 + 1), (5, 64 * 1215 + 7), (3, 64 * 1216 + 1)])
def test_readout_tiles_match_oracle(L, S):
    ebits = inp.random_bits(S, 3 * L ** 3, 0.48, seed=L + S)
    mask = torch.full((S,), 9, dtype=torch.uint8, device=dev())
    counts = torch.full((8,), -5, dtype=torch.int64, device=dev())
    t3d.toric3d_logical(L, S, upload_bits(ebits), mask, counts)
    want = oracle.logical_batch(L, ebits)
    assert np.array_equal(mask.cpu().numpy(), want)
    assert np.array_equal(counts.cpu().numpy(), np.bincount(want, minlength=8))
