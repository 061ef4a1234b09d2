"""Which form a schedule, a run or a batch takes (t3d_column.cu, route_schedule): seen from the kernel
launches counted per kind, where on chip is one launch and step by step one per application, and both
forms' results against each other."""
import pytest
import torch

import paper_2212_06985_gb300 as t3d
import toric3d_inputs as inp
from gpu_util import dev, workspace

pytestmark = pytest.mark.gpu


def count_launches(call, *kinds):
    t3d.toric3d_profile_reset()
    t3d.toric3d_profile_enable(True)
    try:
        call()
    finally:
        t3d.toric3d_profile_enable(False)
    counts = [t3d.toric3d_profile_read(k)[1] for k in kinds]
    t3d.toric3d_profile_reset()
    return counts


def noisy(L, S, p=0.03):
    e = torch.zeros((3 * L ** 3, inp.words_for(S)), dtype=torch.int64, device=dev())
    s = torch.zeros_like(e)
    t3d.toric3d_noise(L, e, p, 5, 0, 1)
    t3d.toric3d_syndrome(L, e, s, p, 5, 0, 1)
    return e, s


@pytest.mark.parametrize("Ls", [[8] * 8, [11, 12, 13, 14, 11, 12, 13, 14], [15, 16, 17, 18, 19, 20, 21, 22]])
def test_small_ensembles_of_a_batch_share_their_launches(Ls):
    # one launch each in series left most of the chip idle: eight ensembles of 1,000 samples took 1.6 to
    # 2.8 times as long as in shared launches
    S, T = 1000, 2
    kw = dict(schedule="FFPFF", n_apply=5, perfect_round=True, perfect_max_sweeps=3)
    items = []
    for i, L in enumerate(Ls):
        e = torch.zeros((3 * L ** 3, inp.words_for(S)), dtype=torch.int64, device=dev())
        items.append(dict(L=L, n_samples=S, sample0=1024 * i, e=e, mask=torch.zeros(S, dtype=torch.uint8, device=dev())))
    batch = t3d.make_batch(items)
    cfg = t3d.make_run_cfg(8, T, 0.03, 0.03, 11, 1, **kw)
    work = workspace(t3d.toric3d_run_batch_workspace_bytes(cfg, batch))
    counts = count_launches(lambda: t3d.toric3d_run_batch(cfg, batch, work), "noise", "syndrome", "pflip")
    assert counts == [T, T + 1, T]   # a schedule of its own would count as p-flip for every item and cycle
    # each ensemble by itself: on chip up to L = 14 wherever that is faster for one
    for item in items:
        L, one = item["L"], t3d.make_run_cfg(item["L"], T, 0.03, 0.03, 11, S, sample0=item["sample0"], **kw)
        e, mask = torch.zeros_like(item["e"]), torch.zeros_like(item["mask"])
        t3d.toric3d_run_cycles(one, e, workspace(t3d.toric3d_run_workspace_bytes(one)), mask)
        assert torch.equal(e, item["e"]) and torch.equal(mask, item["mask"]), L


# step: launches of the step by step form (on chip one launch, three where the columns are turned)
@pytest.mark.parametrize("L,S,schedule,n,step", [(16, 1000, "P", 2, True), (28, 3000, "F", 2, True),
                                                 (26, 20_000, "FFPFF", 5, True), (16, 1000, "F", 8, False),
                                                 (8, 1000, "FFPFF", 5, False), (32, 1000, "FFPFF", 5, False),
                                                 (32, 100_000, "FFPFF", 5, False)])
def test_the_faster_form_of_a_schedule_runs(L, S, schedule, n, step):
    # P P at L = 16, 16 words: 11 us step by step, 43 on chip; F F at L = 28, 48 words 70 and 95; FFPFF at
    # L = 26, 313 words 616 and 756; the others are faster on chip by 1.06 (L = 32, 1,563 words) to 3.6
    e, s = noisy(L, S)
    work = workspace(t3d.toric3d_flip_workspace_bytes(L, e.shape[1]))
    flips, pflips = count_launches(lambda: t3d.toric3d_pflip(L, e, s, schedule, n, 0, 5, 0, 1, work), "flip", "pflip")
    letters = (schedule * n)[:n]
    if step:
        assert (flips, pflips) == (letters.count("F"), letters.count("P"))
    else:
        assert flips + pflips in (1, 3) and flips * pflips == 0


def test_a_lattice_that_fits_runs_whole_on_chip():
    L, S = 8, 1000
    e = torch.zeros((3 * L ** 3, inp.words_for(S)), dtype=torch.int64, device=dev())
    cfg = t3d.make_run_cfg(L, 4, 0.03, 0.03, 11, S, schedule="FFPFF", n_apply=5)
    work = workspace(t3d.toric3d_run_workspace_bytes(cfg))
    assert count_launches(lambda: t3d.toric3d_run_cycles(cfg, e, work), "noise", "syndrome", "pflip") == [0, 0, 0]
