"""gpumcd_plan_open returns while its tally is still being zeroed: a run, a
reset and a result on any stream come after that."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import ledger_exact, make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("how", ["run", "reset", "submit", "result"])
@pytest.mark.parametrize("n_batches", [8, 64])
def test_first_use_on_another_stream(how, n_batches):
    import torch
    ph = W.homogeneous((160, 160, 160), 0.2, W.MAT_WATER, 1.0)
    src = W.pencil(W.ELECTRON, 6.0, 16.0, 16.0)
    ctx = make_ctx()
    pid = ctx.create_phantom(ph)
    side = torch.cuda.Stream()
    d = torch.zeros(ph.nvox, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    doses = []
    for i in range(3):  # the second and third plan reuse a dirty tally
        plan = ctx.plan_open(pid, src, 11, n_batches)
        if how == "result":
            st = ctx.plan_result(plan, 0.5, d.data_ptr(), stream=side.cuda_stream)
            assert st["e_incident"] == 0 and float(d.abs().max()) == 0.0
        if how == "reset":
            ctx.plan_reset(plan, 11, side.cuda_stream)
        if how == "submit":
            ctx.wait(ctx.submit([plan], [640]))
        else:
            ctx.run([plan], [640], side.cuda_stream)
        st = ctx.plan_result(plan, 0.5, d.data_ptr(), stream=side.cuda_stream)
        assert st["e_incident"] == 640 * 6 << 26 and ledger_exact(st)
        doses.append(d.cpu().numpy())
        ctx.plan_close(plan)
    ctx.close()
    assert np.array_equal(doses[0], doses[1]) and np.array_equal(doses[0], doses[2])


def test_reset_in_a_captured_graph():
    """A reset may be captured: its replay zeroes the tally, and the plan stays usable."""
    import torch
    ph = W.homogeneous((16, 16, 16), 0.5, W.MAT_WATER, 1.0)
    src = W.pencil(W.ELECTRON, 6.0, 4.0, 4.0)
    ctx = make_ctx()
    pid = ctx.create_phantom(ph)
    plan = ctx.plan_open(pid, src, 11, 8)
    d = torch.zeros(ph.nvox, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    doses = []
    ctx.run([plan], [640])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.plan_reset(plan, 11, torch.cuda.current_stream().cuda_stream)
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        ctx.run([plan], [640])
        st = ctx.plan_result(plan, 0.5, d.data_ptr())
        assert st["e_incident"] == 640 * 6 << 26 and ledger_exact(st)
        doses.append(d.cpu().numpy())
        ctx.plan_reset(plan, 11)
    ctx.plan_close(plan)
    ctx.close()
    assert np.array_equal(doses[0], doses[1])
