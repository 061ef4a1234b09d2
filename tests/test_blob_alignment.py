"""The training step's weight blob at any 4-byte aligned address (a copy inside a caller's packed buffer): the
convolutions read its rows in 16-byte pieces only where they are 16-byte aligned.  Below 4 bytes the
call returns T3D_EINVAL before anything is launched."""
import ctypes

import pytest
import torch

import cnn_reference as ref
import paper_2212_06985_gb300 as t3d
import toric3d_inputs as inp

EINVAL = 1


@pytest.mark.parametrize("offset", [1, 2, 3, 6])
def test_blob_below_four_bytes_is_refused(offset):
    lib, fake = t3d.lib(), ctypes.c_void_p(0x10000)   # never dereferenced
    status = lib.toric3d_cnn_train_step(4, 64, fake, fake, fake, fake, fake, fake, 1, ctypes.c_float(0.0),
                                        ctypes.c_void_p(0x20000 + offset), None, fake, fake, 1 << 40, None)
    assert status == EINVAL and "blob" in lib.toric3d_last_error().decode()


@pytest.mark.gpu
@pytest.mark.parametrize("offset", [4, 8, 12])
@pytest.mark.parametrize("L,S", [(3, 70), (6, 300)])
def test_training_step_with_a_blob_at_a_four_byte_offset(L, S, offset):
    from gpu_util import dev, upload_bits, workspace
    n, size = 3 * L ** 3, t3d.toric3d_cnn_blob_bytes()
    bits = [upload_bits(inp.random_bits(S, n, 0.1, 7 + k)) for k in range(3)]
    packed = workspace(size + 16)
    results = []
    for at in (0, offset):
        p = torch.from_numpy(ref.random_params(11)).to(dev())
        aligned = workspace(size)
        t3d.toric3d_cnn_prepare(p, aligned)
        blob = packed[at:at + size]
        blob.copy_(aligned)
        m, v, grads = torch.zeros_like(p), torch.zeros_like(p), torch.zeros_like(p)
        loss = torch.zeros(1, dtype=torch.float32, device=dev())
        t3d.toric3d_cnn_train_step(L, S, *bits, p, m, v, 1, 1e-3, blob,
                                   workspace(t3d.toric3d_cnn_train_workspace_bytes(L, S)), loss, grads_out=grads)
        t3d.toric3d_cnn_status()
        t3d.toric3d_cnn_prepare(p, aligned)
        assert torch.equal(blob, aligned[:size])
        results.append((grads.double(), loss.double()))
    # the same arithmetic; the sums reach the gradients by FP32 atomics in any order, at most a few
    # hundred additions each (2^-24 of the running sum an addition)
    for a, b in zip(*results):
        assert float((a - b).norm()) <= 300 * 2 ** -24 * float(a.norm())
