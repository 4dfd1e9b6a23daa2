"""FP64 stream runs of an odd number of steps, whose first step is the one-step
kernel's, against that kernel throughout: out of place, in place, from a graph, keeping
every state, with infinities in the ring."""
import numpy as np
import pytest

from paper_2306_03336_gb300 import j2d5pt, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box", [False, True])
@pytest.mark.parametrize("nx,ny", [(1, 1), (61, 70), (187, 301)])
@pytest.mark.parametrize("steps", [1, 3, 7])
def test_odd_runs(nx, ny, steps, box):
    u = synth.field(nx, ny, 71)
    u[0, nx // 2], u[ny + 1, 0], u[ny // 2 + 1, nx + 1] = np.inf, np.nan, -np.inf
    plan = (j2d5pt.Plan.box9(nx, ny, "f64", synth.box_weights(41)) if box
            else j2d5pt.Plan(nx, ny, "f64", synth.weights(41)))
    src, ref, dst = plan.to_device(u), plan.empty(), plan.empty()
    plan.set("algo", "onestep").run(src, ref, steps)
    plan.sync()
    ref = plan.to_host(ref)
    plan.set("algo", "stream").set("depth", 2)
    for graph in (0, 1):
        plan.set("graph", graph)
        for _ in range(2 + graph):
            dst.zero_()
            plan.run(src, dst, steps)
            plan.sync()
            assert np.array_equal(plan.to_host(dst), ref, equal_nan=True), graph
    plan.set("graph", 0).run(src, src, steps)
    plan.sync()
    assert np.array_equal(plan.to_host(src), ref, equal_nan=True)
    plan.close()


@pytest.mark.parametrize("steps", [1, 3, 7])
def test_odd_kept_states(steps):
    nx, ny = 187, 301
    plan = j2d5pt.Plan(nx, ny, "f64", synth.weights(41))
    src, states = plan.to_device(synth.field(nx, ny, 72)), plan.empty_states(steps)
    plan.set("algo", "stream").set("depth", 2).run_states(src, states, steps)
    plan.set("algo", "onestep")
    for t in range(steps):
        dst = plan.empty()
        plan.run(src, dst, 1)
        plan.sync()
        assert np.array_equal(plan.to_host(states[t]), plan.to_host(dst)), t
        src = dst
    plan.close()
