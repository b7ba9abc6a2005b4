"""A launch sequence that fails after its kernel was enqueued: the call waits for
the stream before it gives the sequence's buffers back (CUDA calls faked on the
host, one of them failing)."""
import pytest

import paper_1101_1245_gb300 as g
import workloads as W
from tests.host_cuda import library


@pytest.fixture
def ctx(monkeypatch):
    L = library()
    L.host_cuda_reset()
    monkeypatch.setattr(g, "_lib", L)
    c = g.engine(0)
    yield c
    L.host_cuda_reset()
    c.close()


@pytest.mark.parametrize("how", ["run", "submit"])
@pytest.mark.parametrize("call", ["cudaMemcpyAsync", "cudaEventRecord", "launch_transport", None])
def test_failed_relaunch_leaves_nothing_pending(ctx, how, call):
    L = library()
    ph = W.homogeneous((4, 4, 4), 0.5, W.MAT_WATER, 1.0)
    pid = ctx.create_phantom(ph)
    plan = ctx.plan_open(pid, W.pencil(W.PHOTON, 6.0, 1.0, 1.0), 1, 8)
    L.host_cuda_leave(2)  # two launches leave records behind: the second relaunch ends the sequence

    def run():
        # the first launch's read-back and event pass, the first relaunch's fails
        nth = {"cudaMemcpyAsync": 3, "cudaEventRecord": 3, "launch_transport": 2}.get(call)
        if how == "run":
            if call:
                L.host_cuda_fail(call.encode(), nth)
            ctx.run([plan], [100])
        else:
            ticket = ctx.submit([plan], [100])
            if call:
                L.host_cuda_fail(call.encode(), 1)
            ctx.wait(ticket)

    if call is None:
        run()
        assert L.host_cuda_calls(b"launch_transport") == 3
    else:
        with pytest.raises(g.GpumcdError) as e:
            run()
        assert e.value.status == g.ERR_CUDA
        assert L.host_cuda_calls(b"launch_transport") == 2
    assert L.host_cuda_pending() == 0
    ctx.plan_close(plan)  # the sequence is settled
