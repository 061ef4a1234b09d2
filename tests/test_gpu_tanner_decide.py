"""A Tanner decode's posteriors and corrections on graphs above the one-kernel iteration's degrees (and, beside
them, on one within), bit for bit the sums of the single iterations' messages in the variables' order: no
iteration, one, several; variables in no check, in up to twelve; ragged batches and chunks."""
import numpy as np
import pytest
import torch

import paper_2212_06985_gb300 as t3d
import toric3d_inputs as inp
from gpu_util import dev, upload_bits, workspace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degree,checks", [(3, 20), (6, 30), (9, 40), (12, 50)])
@pytest.mark.parametrize("S,iters", [(64, 0), (1, 1), (70, 2), (300, 5)])
def test_posteriors_are_the_sums_of_the_messages(degree, checks, S, iters):
    rng = np.random.default_rng(degree + S)
    n = 40
    rows = [sorted(rng.choice(n - 1, degree, replace=False).tolist()) for _ in range(checks)]   # variable n - 1: none
    cptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    cvar = np.array([v for r in rows for v in r], dtype=np.int32)
    g = t3d.tanner_prepare(cptr, cvar, n)
    ebits = (rng.random((S, n)) < 0.1).astype(np.uint8)
    sbits = (rng.random((S, checks)) < 0.3).astype(np.uint8)
    prior = torch.from_numpy(rng.normal(1.0, 1.5, n).astype(np.float32)).to(dev())
    e, s = upload_bits(ebits), upload_bits(sbits)
    llr = torch.empty((n, S), dtype=torch.float32, device=dev())
    t3d.toric3d_tanner_bp(g, S, e, s, prior, iters, workspace(t3d.toric3d_tanner_bp_workspace_bytes(g, S)), llr)

    Sp = 64 * inp.words_for(S)
    msg = [torch.zeros((g.n_edges, Sp), dtype=torch.float32, device=dev()) for _ in range(2)]
    for i in range(iters):
        t3d.toric3d_tanner_bp_step(g, S, upload_bits(sbits), prior, msg[i % 2], msg[(i + 1) % 2], workspace(n * Sp * 4))
    m = msg[iters % 2].cpu().numpy()
    want = np.repeat(prior.cpu().numpy()[:, None], Sp, axis=1)
    for edge, v in enumerate(cvar):   # a variable's edges ascend with its checks
        want[v] = want[v] + m[edge]
    want = want[:, :S]
    assert np.array_equal(llr.cpu().numpy(), want)
    flips = (want < 0).T.astype(np.uint8)
    check = np.zeros((checks, n), dtype=np.uint8)
    for c, r in enumerate(rows):
        check[c, r] = 1
    assert np.array_equal(e.cpu().numpy().view(np.uint64), inp.pack(ebits ^ flips))
    assert np.array_equal(s.cpu().numpy().view(np.uint64), inp.pack(sbits ^ (flips @ check.T & 1)))
    if S > 64 and iters:   # a chunk of one word at a time
        e2, s2 = upload_bits(ebits), upload_bits(sbits)
        t3d.toric3d_tanner_bp(g, S, e2, s2, prior, iters, workspace(t3d.toric3d_tanner_bp_workspace_bytes(g, 64)))
        assert torch.equal(e, e2) and torch.equal(s, s2)
