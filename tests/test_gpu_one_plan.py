"""Launches of one plan run their own kernel (its Philox round keys are kernel
arguments): a plan's tally and sigma are the same bit for bit alone and beside
another plan, on an even and a ragged heterogeneous phantom, for every kernel
that has both forms, and with a captured graph as the count of plans changes."""
import dataclasses

import numpy as np
import pytest

import paper_1101_1245_gb300 as g
import workloads as W
from tests.gpu_common import make_ctx

pytestmark = pytest.mark.gpu

PHANTOMS = {
    "slabs": W.z_slabs((24, 20, 32), 0.5, [(3.0, W.MAT_WATER, 1.0), (2.0, W.MAT_BONE, 1.85),
                                            (4.0, W.MAT_LUNG, 0.26), (1e9, W.MAT_WATER, 1.0)]),
    "ragged": W.smoothed_noise(23, 0.377, np.random.default_rng(2)),
}


def _source(kind, ph):
    X, Y, _ = ph.extent_cm
    if kind == "phsp":
        return dataclasses.replace(W.polyenergetic_phase_space(W.ELECTRON, ph, 501, seed=7),
                                   energy_grouping=W.ENERGY_GROUPED)
    particle = W.ELECTRON if kind == "electron" else W.PHOTON
    return W.Source(particle, W.BEAM_SQUARE, energy=13.0, center_cm=(X / 2, Y / 2), field_cm=4.0)


@pytest.mark.parametrize("flags", [0, g.LAUNCH_GRAPH])
@pytest.mark.parametrize("name", sorted(PHANTOMS))
@pytest.mark.parametrize("kind", ["electron", "photon", "kerma", "phsp"])
def test_alone_equals_beside_another(kind, name, flags):
    import torch
    ph = PHANTOMS[name]
    ctx = make_ctx(flags=flags | (g.LAUNCH_KERMA if kind == "kerma" else 0))
    pid = ctx.create_phantom(ph)
    src = _source(kind, ph)
    plan, other = ctx.plan_open(pid, src, 99, 16), ctx.plan_open(pid, src, 5, 16)
    out = []
    for run in ([plan], [plan, other], [other, plan], [plan]):
        for p in (plan, other):
            ctx.plan_reset(p, 99 if p == plan else 5)
        ctx.run(run, [20_011] * len(run))
        d = torch.zeros(ph.nvox, dtype=torch.float64, device="cuda")
        s = torch.zeros_like(d)
        ctx.plan_result(plan, 0.5, d.data_ptr(), s.data_ptr())
        out.append((d.cpu().numpy(), s.cpu().numpy()))
    ctx.close()
    for d, s in out[1:]:
        assert np.array_equal(d, out[0][0]) and np.array_equal(s, out[0][1])
