"""toric3d_bp's workspace holds 32-byte records behind message buffers of whole multiples of 32 bytes, so
an address that is only 8- or 16-byte aligned is refused before anything is launched."""
import ctypes

import pytest

import paper_2212_06985_gb300 as t3d

EINVAL = 1


@pytest.mark.parametrize("offset", [8, 16, 48])
@pytest.mark.parametrize("iters", [0, 1, 2])
def test_workspace_below_32_bytes_is_refused(offset, iters):
    lib, fake = t3d.lib(), ctypes.c_void_p(0x10000)   # never dereferenced
    status = lib.toric3d_bp(4, 10, fake, fake, 0.1, 0.1, iters, ctypes.c_void_p(0x20000 + offset), 1 << 30, None, None)
    assert status == EINVAL and "32-byte aligned" in lib.toric3d_last_error().decode()


def test_message_buffers_keep_the_alignment():
    for L in (2, 3, 5, 128):
        for n in (1, 64, 65):
            assert t3d.toric3d_bp_message_bytes(L, n) % 32 == 0
