"""The energy-grouping sort at the edges of its blocks and of its two block
sizes: every history is claimed once, so the grouped tally equals the
ungrouped one bit for bit (phase spaces: one kernel runs both)."""
import dataclasses

import numpy as np
import pytest

import workloads as W
from tests.gpu_common import make_ctx
from tests.test_gpu_repro import EVENT_KEYS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 255, 1023, 1024, 1025, (1 << 19) - 1, 1 << 19, (1 << 19) + 1])
def test_grouped_equals_ungrouped(n):
    import torch
    ph = W.homogeneous((6, 6, 6), 0.5, W.MAT_WATER, 1.0)
    src = W.polyenergetic_phase_space(W.PHOTON, ph, 777, seed=3)
    ctx = make_ctx()
    pid = ctx.create_phantom(ph)
    got = []
    for grouping in (W.ENERGY_UNGROUPED, W.ENERGY_GROUPED):
        plan = ctx.plan_open(pid, dataclasses.replace(src, energy_grouping=grouping), 5, 8)
        ctx.run([plan], [n])
        d = torch.zeros(ph.nvox, dtype=torch.float64, device="cuda")
        st = ctx.plan_result(plan, 0.5, d.data_ptr())
        got.append((d.cpu().numpy(), [st[k] for k in EVENT_KEYS]))
        ctx.plan_close(plan)
    ctx.close()
    assert np.array_equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
