"""Replay of a sequence's first launch from a captured graph (GPUMCD_LAUNCH_GRAPH),
with CUDA calls faked on the host: what each replay hands the kernel."""
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
