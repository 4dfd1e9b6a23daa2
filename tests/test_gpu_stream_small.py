"""Stream passes on small grids (several warps to a run, passes launched before the
one they follow has ended) against the one-step kernel, bit for bit: ragged sizes,
runs in place, several runs in a row on a side stream, and graph replay."""
import numpy as np
import pytest

from paper_2306_03336_gb300 import j2d5pt, synth

pytestmark = pytest.mark.gpu


def reference(u, w, nx, ny, dt, steps):
    plan = j2d5pt.Plan(nx, ny, dt, w).set("algo", "onestep")
    src, dst = plan.to_device(u), plan.empty()
    plan.run(src, dst, steps)
    plan.sync()
    got = plan.to_host(dst)
    plan.close()
    return got


@pytest.mark.parametrize("dt,box", [("f64", False), ("f32", False), ("f32", True)])
@pytest.mark.parametrize("nx,ny", [(1, 1), (5, 40), (113, 21), (112, 22), (449, 317), (1000, 83)])
def test_auto_small_grids(nx, ny, dt, box):
    u = synth.field(nx, ny, 11)
    w = synth.box_weights(12) if box else synth.weights(12)
    for steps in (4, 13):
        ref = reference(u, w, nx, ny, dt, steps)
        for algo in ("auto", "stream"):
            plan = j2d5pt.Plan(nx, ny, dt, w).set("algo", algo)
            src, dst = plan.to_device(u), plan.empty()
            plan.run(src, dst, steps)
            plan.run(src, src, steps)
            plan.sync()
            assert np.array_equal(plan.to_host(dst), ref), (algo, steps)
            assert np.array_equal(plan.to_host(src), ref), (algo, steps, "in place")
            plan.close()


@pytest.mark.parametrize("dt", ["f64", "f32"])
def test_chained_runs_and_graph(dt):
    import torch
    nx, ny, steps = 300, 217, 10
    u, w = synth.field(nx, ny, 21), synth.weights(22)
    ref = reference(u, w, nx, ny, dt, 3 * steps)
    side = torch.cuda.Stream()
    for graph in (0, 1):
        plan = j2d5pt.Plan(nx, ny, dt, w).set("algo", "stream").set("graph", graph)
        a, b = plan.to_device(u), plan.empty()
        first = a.clone()
        torch.cuda.synchronize()
        for rep in range(3):
            with torch.cuda.stream(side):
                a.copy_(first)
                plan.run(a, b, steps, stream=side)
                plan.run(b, a, steps, stream=side)
                plan.run(a, b, steps, stream=side)
                got = b.clone()
            side.synchronize()
            assert np.array_equal(plan.to_host(got), ref), (graph, rep)
        plan.close()
