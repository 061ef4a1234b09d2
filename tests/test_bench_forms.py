"""Which form of a schedule the flip / p-flip roofline sees in the launches recorded per kind: step by step an
application is one record, whatever its letter; on chip the whole schedule is one record, or three
where its columns are turned, all of one kind."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _roofline(flip, pflip, steps, **changes):
    sys.path.insert(0, ROOT)
    import dataclasses
    import bench
    import toric3d_inputs as inp
    w = dataclasses.replace(inp.WORKLOADS["pflip_L32"], **changes)
    prof = {k: (0.0, 0) for k in ("noise", "syndrome", "flip", "pflip", "bp_step", "bp_decide", "logical", "layout",
                                  "cnn")}
    prof.update(noise=(1.8 * steps, steps), syndrome=(2.0 * steps, steps), flip=flip, pflip=pflip)
    return bench.sweep_roofline(prof, w, inp.n_bits(32), 100_000, steps, 10.0 * steps, 6780.0, "test", {"sm_mhz": 2070.0})


@pytest.mark.parametrize("steps", [1, 4])
def test_step_by_step(steps):
    # F F P F F: four flip records and one p-flip record a cycle
    r = _roofline((3.6 * steps, 4 * steps), (1.6 * steps, steps), steps)
    assert r["kernel"] == "k_flip_tiled" and abs(r["ms_per_application"] - 0.9) < 1e-9
    assert set(r["kernels_hbm_frac"]) == {"noise", "syndrome", "flip", "pflip"}


@pytest.mark.parametrize("records", [1, 3])
@pytest.mark.parametrize("steps", [1, 4])
def test_on_chip(records, steps):
    r = _roofline((0.0, 0), (5.2 * steps, records * steps), steps)
    assert r["kernel"].startswith("k_slab") and abs(r["ms_per_application"] - 5.2) < 1e-9
    r = _roofline((0.0, 0), (5.2 * steps, records * steps), steps, schedule="FFP", n_apply=3)
    assert r["kernel"].startswith("k_slab")
