"""A captured graph (GPUMCD_LAUNCH_GRAPH) after other materials were loaded: the
replayed kernel's shared memory holds their tables, and the dose is a direct
launch's."""
import numpy as np
import pytest

import paper_1101_1245_gb300 as g
import workloads as W
from tests.gpu_common import make_ctx

pytestmark = pytest.mark.gpu


def test_replay_after_loading_more_materials():
    ph = W.z_slabs((12, 12, 16), 0.5, [(2.0, W.MAT_WATER, 1.0), (2.0, W.MAT_BONE, 1.85), (1e9, W.MAT_LUNG, 0.26)])
    water = W.homogeneous((12, 12, 16), 0.5, W.MAT_WATER, 1.0)
    src = W.Source(W.ELECTRON, W.BEAM_SQUARE, energy=9.0, center_cm=(3.0, 3.0), field_cm=4.0)
    doses = []
    for flags in (0, g.LAUNCH_GRAPH):
        ctx = make_ctx(flags=flags)
        for n, p in ((1, water), (len(W.MATERIALS), ph), (1, water)):
            ctx.load_materials(W.MATERIALS[:n], W.DEFAULT_PHYSICS)
            pid = ctx.create_phantom(p)
            r = ctx.simulate(pid, src, 20_000, 3, nvox=p.nvox)
            doses.append(r.dose)
            ctx.destroy_phantom(pid)
        ctx.close()
    for a, b in zip(doses[:3], doses[3:]):
        assert np.array_equal(a, b)
