"""AUTO with a depth the caller set: every depth that the tiles, the skewed tiles and
the resident kernel take runs, whatever schedule AUTO prefers without one, and gives
the one-step kernel's cells bit for bit."""
import numpy as np
import pytest

from paper_2306_03336_gb300 import j2d5pt, synth

pytestmark = pytest.mark.gpu


def plan_of(nx, ny, dt, box):
    if box:
        return j2d5pt.Plan.box9(nx, ny, dt, synth.box_weights(41))
    return j2d5pt.Plan(nx, ny, dt, synth.weights(41))


@pytest.mark.parametrize("nx,ny,dt,box", [(200, 120, "f32", False), (2304, 1700, "f64", False), (130, 203, "f64", True),
                                          (130, 203, "f32", True)])
def test_auto_with_a_depth(nx, ny, dt, box):
    import torch
    one = plan_of(nx, ny, dt, box).set("algo", "onestep")
    u = synth.field(nx, ny, 42)
    src, ref, got = one.to_device(u.astype(np.float32) if dt == "f32" else u), one.empty(), one.empty()
    for steps in (5, 6, 13):
        one.run(src, ref, steps)
        one.sync()
        for depth in (0, 2, 3, 4, 5, 6, 8, 12, 16):
            if dt == "f64" and not box and depth > 8:
                continue
            p = plan_of(nx, ny, dt, box).set("depth", depth)
            got.zero_()
            p.run(src, got, steps)
            p.sync()
            assert torch.equal(p.view(got), one.view(ref)), (steps, depth)
            p.close()
    one.close()


@pytest.mark.parametrize("nx,ny,dt,box,routes", [
    (200, 120, "f32", False, {0: "stream", 2: "resident", 4: "stream", 5: "resident", 8: "stream", 10: "resident", 16: "resident"}),
    (2304, 1700, "f64", False, {0: "stream", 2: "stream", 3: "tiles", 4: "tiles", 6: "tiles", 8: "tiles"}),
    (130, 203, "f64", True, {0: "stream", 2: "stream", 3: "skewed", 4: "skewed", 8: "skewed"}),
    (130, 203, "f32", True, {0: "stream", 4: "stream", 8: "stream", 10: "skewed", 16: "skewed"})])
def test_auto_route_of_a_depth(nx, ny, dt, box, routes):
    for depth, algo in routes.items():
        p = plan_of(nx, ny, dt, box).set("depth", depth)
        assert "algo=%s " % algo in p.describe(), (depth, p.describe())
        p.close()
