"""Replay of a sequence's first launch from a captured graph (GPUMCD_LAUNCH_GRAPH),
with CUDA calls faked on the host: what each replay hands the kernel."""
import ctypes as C

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
    c.set_launch(flags=g.LAUNCH_GRAPH)
    yield c
    c.close()


def open_plan(ctx):
    pid = ctx.create_phantom(W.homogeneous((4, 4, 4), 0.5, W.MAT_WATER, 1.0))
    return pid, ctx.plan_open(pid, W.pencil(W.PHOTON, 6.0, 1.0, 1.0), 1, 8)


def test_shared_memory_follows_the_loaded_materials(ctx):
    """Materials may be loaded again once no phantom uses them: a graph captured
    with the tables of one material launches with those of three."""
    L = library()
    for n in (1, len(W.MATERIALS), 2):
        ctx.load_materials(W.MATERIALS[:n], W.DEFAULT_PHYSICS)
        pid, plan = open_plan(ctx)
        ctx.run([plan], [100])
        ctx.plan_close(plan)
        ctx.destroy_phantom(pid)
    assert L.host_cuda_calls(b"cudaGraphLaunch") == 3
    assert L.host_cuda_misfits() == 0


def test_alternating_kernels_are_captured_once(ctx):
    """One plan and several run different compiled kernels: runs that alternate
    rewrite arguments and capture nothing after each kernel's first run."""
    L = library()
    pid, a = open_plan(ctx)
    _, b = open_plan(ctx)
    for _ in range(5):
        ctx.run([a], [100])
        ctx.run([a, b], [100, 100])
    assert L.host_cuda_calls(b"cudaGraphLaunch") == 10
    assert L.host_cuda_calls(b"cudaGraphInstantiate") == 2
    fn = (C.c_void_p * 10)()
    assert L.host_cuda_launched(fn, 10) == 10
    assert len({fn[i] for i in range(0, 10, 2)}) == len({fn[i] for i in range(1, 10, 2)}) == 1
    assert fn[0] != fn[1]


def test_another_launch_shape_is_captured_again(ctx):
    L = library()
    _, a = open_plan(ctx)
    for threads in (1024, 512, 512, 1024):
        ctx.set_launch(block_threads=threads, flags=g.LAUNCH_GRAPH)
        ctx.run([a], [100])
    assert L.host_cuda_calls(b"cudaGraphInstantiate") == 3
    assert L.host_cuda_calls(b"cudaGraphExecDestroy") == 2


@pytest.mark.parametrize("call", ["cudaStreamBeginCapture", "cudaGraphInstantiate", "cudaGraphGetNodes",
                                  "cudaGraphExecKernelNodeSetParams", "cudaGraphLaunch"])
def test_a_failed_capture_is_reported_and_tried_again(ctx, call):
    L = library()
    _, a = open_plan(ctx)
    if call == "cudaGraphExecKernelNodeSetParams":
        ctx.run([a], [100])
    L.host_cuda_fail(call.encode(), 1)
    with pytest.raises(g.GpumcdError) as e:
        ctx.run([a], [100])
    assert e.value.status == g.ERR_CUDA and L.host_cuda_pending() == 0
    ctx.plan_reset(a, 1)
    ctx.run([a], [100])
    assert ctx.plan_histories(a) == 100
