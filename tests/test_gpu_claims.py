"""Claims of primaries: a warp takes a share of a source that depends on the
histories left.  Every history runs once whatever the counts: at the edges of
a grid's warps and of a chunk per warp, the tally and every counter equal those
of the same histories run in single-chunk pieces."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import make_ctx
from tests.test_gpu_repro import EVENT_KEYS

pytestmark = pytest.mark.gpu

WARPS = 152 * 32  # of the default launch on the chip


def _run(ctx, ph, src, parts):
    import torch
    pid = ctx.create_phantom(ph)
    plan = ctx.plan_open(pid, src, 5, 8)
    for n in parts:
        ctx.run([plan], [n])
    d = torch.zeros(ph.nvox, dtype=torch.float64, device="cuda")
    st = ctx.plan_result(plan, 0.5, d.data_ptr())
    ctx.plan_close(plan)
    ctx.destroy_phantom(pid)
    return d.cpu().numpy(), [st[k] for k in EVENT_KEYS]


@pytest.mark.parametrize("n", [1, 31, WARPS - 1, WARPS, WARPS + 1, 2 * WARPS - 1, 32 * WARPS - 1, 32 * WARPS + 1])
@pytest.mark.parametrize("particle", [W.PHOTON, W.ELECTRON])
def test_every_history_is_claimed_once(n, particle):
    ph = W.homogeneous((6, 6, 6), 0.5, W.MAT_WATER, 1.0)
    src = W.Source(particle, W.BEAM_SQUARE, energy=1.0, center_cm=(1.5, 1.5), field_cm=2.0)
    ctx = make_ctx()
    whole, counts = _run(ctx, ph, src, [n])
    assert counts[0] == n << 26  # incident: 1 MeV is 2^26 quanta
    parts = [n // 3, n - n // 3] if n > 2 else [n]
    ctx.set_launch(chunk=7)
    split, split_counts = _run(ctx, ph, src, parts)
    ctx.close()
    assert np.array_equal(whole, split)
    assert counts == split_counts
