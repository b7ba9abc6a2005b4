"""The cycle profile counts every electron step as a pass: the active lanes of its
electron passes sum to the steps taken."""
import pytest

import paper_1101_1245_gb300 as g
import workloads as W
from tests.gpu_common import make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("particle", [W.PHOTON, W.ELECTRON])
@pytest.mark.parametrize("n", [7, 20_000])
def test_electron_lanes_are_the_steps(particle, n):
    ph = W.z_slabs((24, 20, 32), 0.5, [(3.0, W.MAT_WATER, 1.0), (1e9, W.MAT_LUNG, 0.26)])
    src = W.Source(particle, W.BEAM_SQUARE, energy=9.0, center_cm=(6.0, 5.0), field_cm=4.0)
    ctx = make_ctx(flags=g.LAUNCH_PROFILE)
    pid = ctx.create_phantom(ph)
    plan = ctx.plan_open(pid, src, 5, 8)
    ctx.run([plan], [n])
    st = ctx.plan_result(plan, 0.5)
    pr = ctx.profile()["electron"]
    lanes = pr["lane_occupancy"] * 32 * pr["iterations"]
    ctx.close()
    assert round(lanes) == st["n_electron_steps"] > 0
    assert 0 < pr["lane_occupancy"] <= 1
