"""BP's first two iterations in one launch (toric3d_bp) against the same iterations one by one
(toric3d_bp_step): the posteriors equal bit for bit, for one to four iterations, with and without
measurement-error variables, on lattices where every neighbour wraps (L = 2, 3) and larger ones,
ragged batches, chunked and whole."""
import pytest
import torch

import paper_2212_06985_gb300 as t3d
import toric3d_inputs as inp
from gpu_util import dev, upload_bits, workspace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q", [0.0, 0.04])
@pytest.mark.parametrize("L,S", [(2, 70), (3, 64), (5, 130), (8, 1)])
@pytest.mark.parametrize("iters", [1, 2, 3, 4])
def test_decode_equals_single_iterations(L, S, iters, q):
    n = 3 * L ** 3
    s = upload_bits(inp.random_bits(S, n, 0.2, seed=L + S))
    e = torch.zeros_like(s)
    msg = [torch.empty(t3d.toric3d_bp_message_bytes(L, S) // 4, dtype=torch.float32, device=dev()) for _ in range(2)]
    for k in range(iters):
        t3d.toric3d_bp_step(L, S, s, 0.04, q, msg[(k + 1) % 2] if k else None, msg[k % 2])
    want = torch.empty((n, S), dtype=torch.float32, device=dev())
    we, ws = e.clone(), s.clone()
    t3d.toric3d_bp_decide(L, S, msg[(iters - 1) % 2], 0.04, we, ws,
                          workspace(t3d.toric3d_bp_decide_workspace_bytes(L, S)), want)
    got = torch.empty_like(want)
    ge, gs = e.clone(), s.clone()
    t3d.toric3d_bp(L, S, ge, gs, 0.04, q, iters, workspace(t3d.toric3d_bp_workspace_bytes(L, S)), got)
    assert torch.equal(got, want) and torch.equal(ge, we) and torch.equal(gs, ws)
    ge, gs = e.clone(), s.clone()
    t3d.toric3d_bp(L, S, ge, gs, 0.04, q, iters, workspace(t3d.toric3d_bp_workspace_bytes(L, 64)))
    assert torch.equal(ge, we) and torch.equal(gs, ws)
