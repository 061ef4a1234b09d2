"""The weight gradients' column walk against the FP32 PyTorch CPU reference, layer by layer: lattices
where a row is shorter than the rings (L = 2, 3) and longer, odd and even, one sample tile and
several, the last one partly padding, fewer rows than thread blocks and several rows a block."""
import numpy as np
import pytest
import torch

import cnn_reference as ref
import paper_2212_06985_gb300 as t3d
import toric3d_inputs as inp
from gpu_util import dev, upload_bits, workspace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,S", [(2, 70), (3, 129), (7, 130), (8, 64), (10, 300), (9, 700)])
def test_every_layers_gradient_matches_reference(L, S):
    n = 3 * L ** 3
    params = ref.random_params(40 + L)
    sp = inp.random_bits(S, n, 0.15, 1 + L)
    sc = inp.random_bits(S, n, 0.15, 2 + L)
    y = inp.random_bits(S, n, 0.08, 3 + L)
    p = torch.from_numpy(params).to(dev())
    blob = workspace(t3d.toric3d_cnn_blob_bytes())
    t3d.toric3d_cnn_prepare(p, blob)
    m, v, grads = torch.zeros_like(p), torch.zeros_like(p), torch.zeros_like(p)
    loss = torch.zeros(1, dtype=torch.float32, device=dev())
    t3d.toric3d_cnn_train_step(L, S, upload_bits(sp), upload_bits(sc), upload_bits(y), p, m, v, 1, 0.0, blob,
                               workspace(t3d.toric3d_cnn_train_workspace_bytes(L, S)), loss, grads_out=grads)
    torch.cuda.synchronize()
    t3d.toric3d_cnn_status()
    _, want = ref.loss_and_grad(params, L, sp, sc, y)
    got, want = ref.unpack(grads.cpu().numpy()), ref.unpack(want)
    # the kernels round activations, weights and gradients to BF16 at up to six places on the way to
    # a layer (2^-9 each, 1.2%), and the gates of as many pre-activations lie that close to zero
    for name, _ in ref.SIZES:
        err = float((got[name] - want[name]).norm() / want[name].norm())
        print(f"{name} relative error {err:.3e}")
        assert err < 0.05, name
