"""The noise's six high bits over thresholds with every kind of bit pair (blocks of two zero bits are
compared at once), against the oracle, bit for bit: one site and many sites per thread."""
import numpy as np
import pytest

import oracle
import paper_2212_06985_gb300 as t3d
from gpu_util import download_bits, zeros_words

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [0.5 / 64, 1 / 64, 0.02, 3.5 / 64, 1 / 16, 0.0817, 0.15, 0.25, 0.2655, 0.26, 0.5, 0.77])
@pytest.mark.parametrize("L,S", [(3, 70), (16, 64 * 40)])
def test_noise_of_every_rate_matches_oracle(L, S, p):
    e = zeros_words(3 * L ** 3, S)
    t3d.toric3d_noise(L, e, p, 21, 64, 5)
    got = download_bits(e, S)
    k = min(S, 70)
    start = np.zeros((k, 3 * L ** 3), dtype=np.uint8)
    assert np.array_equal(got[:k], oracle.noise_batch(L, start, p, 21, 64, 5))
    assert abs(got.mean() - p) < 6 * np.sqrt(p * (1 - p) / got.size)
