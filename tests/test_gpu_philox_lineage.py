"""The transport keeps what the first two Philox rounds make of a particle's
lineage instead of the lineage: its draws equal Philox4x32-10 of the counter
(draw, lineage lo, lineage hi, history), for keys and histories at the ends of
their ranges."""
import numpy as np
import pytest

from tests.gpu_common import make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [0, 1, 0xFFFFFFFF, 0x9E3779B97F4A7C15, (1 << 64) - 1])
def test_draws_equal_philox(seed):
    n = 4099
    ctx = make_ctx()
    # past 20 transport mean free paths the multiple-scattering sampler returns
    # its uniform, (top 24 bits of the third word + 1) 2^-24; history i's first
    # draw has lineage (i >> 32, 0x5EED)
    got = ctx.debug_sample(4, 25.0, n, seed)
    ctr = np.zeros((n, 4), dtype=np.uint32)
    ctr[:, 2] = 0x5EED
    ctr[:, 3] = np.arange(n)
    w = ctx.debug_philox(ctr, [seed & 0xFFFFFFFF, seed >> 32], use_curand=True)[:, 2]
    ctx.close()
    assert np.array_equal(got, ((w >> 8).astype(np.float64) + 1.0).astype(np.float32) * np.float32(2.0 ** -24))
