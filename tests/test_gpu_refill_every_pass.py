"""The ablation's pool (GPUMCD_REFILL_EVERY_PASS) runs the kernel of the other
refill policies, one electron step a pass: the same tally and counters as the
default launch, and the value of the header."""
import re

import numpy as np
import pytest

import paper_1101_1245_gb300 as g
import workloads as W
from tests.gpu_common import make_ctx
from tests.test_abi import HEADER
from tests.test_gpu_repro import EVENT_KEYS


def test_value_matches_the_header():
    m = re.search(r"^#define GPUMCD_REFILL_EVERY_PASS (0x[0-9A-Fa-f]+)u", open(HEADER).read(), flags=re.M)
    assert m and int(m.group(1), 16) == g.REFILL_EVERY_PASS


@pytest.mark.gpu
@pytest.mark.parametrize("particle", [W.PHOTON, W.ELECTRON])
@pytest.mark.parametrize("n", [5, 40_000])
def test_bit_identical_to_the_default(particle, n):
    ph = W.z_slabs((24, 20, 32), 0.5, [(3.0, W.MAT_WATER, 1.0), (2.0, W.MAT_BONE, 1.85), (1e9, W.MAT_LUNG, 0.26)])
    src = W.Source(particle, W.BEAM_SQUARE, energy=13.0, center_cm=(6.0, 5.0), field_cm=4.0)
    out = []
    for launch in ({}, dict(refill_period=g.REFILL_EVERY_PASS),
                   dict(refill_period=g.REFILL_EVERY_PASS, block_threads=256, blocks_per_sm=2)):
        ctx = make_ctx(**launch)
        pid = ctx.create_phantom(ph)
        out.append(ctx.simulate(pid, src, n, 9, nvox=ph.nvox))
        ctx.close()
    for r in out[1:]:
        assert np.array_equal(r.dose, out[0].dose) and np.array_equal(r.sigma, out[0].sigma)
        assert all(r.stats[k] == out[0].stats[k] for k in EVENT_KEYS)
