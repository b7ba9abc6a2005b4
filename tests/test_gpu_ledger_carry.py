"""The per-CTA ledgers are a 32-bit low word with a carry: sums at and around
2^32 quanta (64 MeV) come out exact, for every lane count that adds at once."""
import pytest

import workloads as W
from tests.gpu_common import ledger_exact, make_ctx

pytestmark = pytest.mark.gpu


# 16 MeV is 2^30 quanta: four histories reach 2^32 exactly
@pytest.mark.parametrize("n", [1, 3, 4, 5, 31, 32, 33, 1000, 40_001])
@pytest.mark.parametrize("particle", [W.PHOTON, W.ELECTRON])
def test_escaped_and_incident_energy_are_exact(n, particle):
    ph = W.homogeneous((4, 4, 4), 0.5, W.MAT_WATER, 1.0)
    outside = W.pencil(particle, 16.0, -1.0, -1.0)  # misses the phantom: all of it escapes
    inside = W.pencil(particle, 16.0, 1.0, 1.0)
    ctx = make_ctx()
    pid = ctx.create_phantom(ph)
    for src in (outside, inside):
        st = ctx.simulate(pid, src, n, 3, nvox=ph.nvox).stats
        assert st["e_incident"] == n << 30
        assert ledger_exact(st)
        if src is outside:
            assert st["e_escaped"] == n << 30
    ctx.close()
