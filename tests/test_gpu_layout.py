"""Layout conversion (toric3d_pack / toric3d_unpack) at the edges of its tiles: column counts
around 128 and words around 16 per block, rows that are and are not 4-byte aligned (odd n_bits, a
bits array that starts at an odd address), byte values other than 0 / 1 (only bit 0 counts)."""
import numpy as np
import pytest
import torch

import paper_2212_06985_gb300 as t3d
import toric3d_inputs as inp
from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("n,S", [(1, 65), (3, 64), (4, 1), (127, 130), (128, 1024), (129, 1025), (256, 1088),
                                 (260, 2049), (192, 63), (81, 5000)])
def test_pack_and_unpack_tiles(n, S, offset):
    rng = np.random.default_rng(n + S)
    raw = rng.integers(0, 256, (S, n), dtype=np.uint8)
    W = inp.words_for(S)
    room = torch.full((S * n + 8,), 0xAA, dtype=torch.uint8, device=dev())
    bits = room[offset:offset + S * n].view(S, n)
    bits.copy_(torch.from_numpy(raw))
    words = torch.full((n + 2, W), -1, dtype=torch.int64, device=dev())
    t3d.toric3d_pack(n, S, bits, words[1:n + 1])
    assert np.array_equal(words[1:n + 1].cpu().numpy().view(np.uint64), inp.pack(raw & 1))
    assert int(words[0].min()) == int(words[0].max()) == int(words[n + 1].min()) == int(words[n + 1].max()) == -1
    bits.fill_(0xAA)
    t3d.toric3d_unpack(n, S, words[1:n + 1], bits)
    assert np.array_equal(bits.cpu().numpy(), raw & 1)
    rest = torch.cat([room[:offset], room[offset + S * n:]])
    assert int(rest.min()) == int(rest.max()) == 0xAA       # nothing beside the array is written
