"""The weight gradients tap by tap against the same sums in FP64, with the kernels' BF16 rounding points in the
backward pass too (the gradients at the three pre-activations), so that what is left is the FP32
accumulation and the few values whose rounding it turns."""
import numpy as np
import pytest
import torch

import cnn_reference as ref
import paper_2212_06985_gb300 as t3d
import toric3d_inputs as inp
from gpu_util import dev, upload_bits, workspace

pytestmark = pytest.mark.gpu

TAPS = [(z, y, x) for z in range(3) for y in range(3) for x in range(3)]


def _weight_grad(x, d):
    g = torch.zeros(d.shape[1], x.shape[1], 3, 3, 3, dtype=torch.float64)
    for k in TAPS:
        g[:, :, k[0], k[1], k[2]] = torch.einsum("sizyx,sozyx->oi", torch.roll(x, [1 - v for v in k], (2, 3, 4)), d)
    return g


def _data_grad(d, w):
    return sum(torch.einsum("sozyx,oi->sizyx", torch.roll(d, [v - 1 for v in k], (2, 3, 4)), w[:, :, k[0], k[1], k[2]])
               for k in TAPS)


def _gradients(params, L, sp, sc, y):
    P = {k: v.double() for k, v in ref.unpack(params).items()}
    W = {k: ref.bf16(v.float()).double() for k, v in P.items() if k in ("w1", "w2", "w3")}
    rnd = lambda v: ref.bf16(v.float()).double()
    b = lambda v: v.view(1, -1, 1, 1, 1)
    x = ref.features(L, sp, sc).double()
    h1 = rnd(torch.relu(ref._conv(x, W["w1"]) + b(P["b1"])))
    h2 = rnd(torch.relu(ref._conv(h1, W["w2"]) + b(P["b2"])))
    h3 = torch.relu(ref._conv(h2, W["w3"]) + b(P["b3"]))
    z = torch.einsum("sczyx,dc->sdzyx", h3, P["w4"]) + b(P["b4"])
    dz = (torch.sigmoid(z) - torch.from_numpy(y.reshape(z.shape).astype(np.float64))) / z.numel()
    d3 = rnd((h3 > 0) * torch.einsum("sdzyx,dc->sczyx", dz, P["w4"]))
    d2 = rnd((h2 > 0) * _data_grad(d3, W["w3"]))
    d1 = rnd((h1 > 0) * _data_grad(d2, W["w2"]))
    return {"w3": _weight_grad(h2, d3), "w2": _weight_grad(h1, d2), "w1": _weight_grad(x, d1)}


@pytest.mark.parametrize("L,S", [(2, 70), (3, 129), (7, 130), (8, 64), (9, 200)])
def test_every_taps_gradient_matches_the_same_sums(L, S):
    n = 3 * L ** 3
    params = ref.random_params(40 + L)
    sp, sc, y = (inp.random_bits(S, n, q, k + L) for q, k in ((0.15, 1), (0.15, 2), (0.08, 3)))
    p = torch.from_numpy(params).to(dev())
    blob = workspace(t3d.toric3d_cnn_blob_bytes())
    t3d.toric3d_cnn_prepare(p, blob)
    m, v, grads = torch.zeros_like(p), torch.zeros_like(p), torch.zeros_like(p)
    loss = torch.zeros(1, dtype=torch.float32, device=dev())
    t3d.toric3d_cnn_train_step(L, S, upload_bits(sp), upload_bits(sc), upload_bits(y), p, m, v, 1, 0.0, blob,
                               workspace(t3d.toric3d_cnn_train_workspace_bytes(L, S)), loss, grads_out=grads)
    torch.cuda.synchronize()
    t3d.toric3d_cnn_status()
    got = ref.unpack(grads.cpu().numpy())
    # FP32 sums are about 2^-20 off, which turns the BF16 rounding (one unit, 2^-8) of about 2^-20 / 2^-8 = 2^-12 of
    # the values a layer on: 2^-8 sqrt(2^-12) = 2^-14 of a sum of random terms, and as much again for each of the
    # three layers behind it; four times that
    for name, want in _gradients(params, L, sp, sc, y).items():
        err = (got[name].double() - want).flatten(2).norm(dim=(0, 1)) / want.flatten(2).norm(dim=(0, 1))
        print(f"{name} largest tap error {float(err.max()):.2e}")
        assert float(err.max()) < 2 ** -10, name
