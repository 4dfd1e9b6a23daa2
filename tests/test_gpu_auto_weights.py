"""What AUTO makes of a plan's FP64 weights: a window (windowed fixed point), positive
without a window, or cells that are chains throughout; and that the schedule it takes
gives the one-step kernel's cells bit for bit."""
import numpy as np
import pytest

from paper_2306_03336_gb300 import j2d5pt, synth

pytestmark = pytest.mark.gpu

TINY = float(np.finfo(np.float64).tiny)
FIVE = [  # weights, int_path, schedule of a grid too large for the chip
    ([0.5, 0.25, 0.04, 0.15, 0.06], 1, "stream"),
    ([0.55, 0.2, 0.0005, 0.1395, 0.11], 1, "tiles"),
    ([0.55, 0.2, 2.0 ** -11, 0.13, 0.11], 1, "tiles"),
    ([0.55, 0.2, 0.99 * 2.0 ** -11, 0.13, 0.11], 1, "stream"),
    ([0.55, 0.2, TINY, 0.13, 0.11], 1, "stream"),
    ([0.55, 0.2, TINY / 2, 0.13, 0.11], 1, "stream"),
    ([0.25, 0.25, 0.25, 0.0, 0.25], 1, "stream"),
    ([0.3, 0.3, -0.1, 0.25, 0.25], 1, "stream"),
    ([0.55, 0.2, 0.0005, 0.1395, 0.11], 0, "stream"),
]


@pytest.mark.parametrize("w,path,algo", FIVE)
def test_five_point_route(w, path, algo):
    import torch
    nx, ny, steps = 2304, 1700, 7
    p = j2d5pt.Plan(nx, ny, "f64", np.array(w)).set("int_path", path)
    assert "algo=%s " % algo in p.describe(), p.describe()
    src, got, ref = p.to_device(synth.field(nx, ny, 51)), p.empty(), p.empty()
    p.run(src, got, steps)
    p.set("algo", "onestep").run(src, ref, steps)
    p.sync()
    assert torch.equal(p.view(got), p.view(ref))
    p.close()


def test_large_grids_and_short_spreads_keep_the_stream():
    w = np.array([0.55, 0.2, 0.0005, 0.1395, 0.11])
    p = j2d5pt.Plan(8192, 8192, "f64", w)
    assert "algo=stream " in p.describe()
    p.close()


@pytest.mark.parametrize("nx,ny,w,launches", [
    (2304, 1700, FIVE[0][0], 8),  # below 8 M cells: the one-step kernel
    (4096, 2100, FIVE[0][0], 4),  # a window: passes of two steps
    (4096, 2100, FIVE[1][0], 8),  # positive without a window
    (4096, 2100, FIVE[4][0], 8)])  # a zero weight
def test_kept_states_route(nx, ny, w, launches):
    import torch
    steps = 8
    p = j2d5pt.Plan(nx, ny, "f64", np.array(w))
    src, one = p.to_device(synth.field(nx, ny, 52)), p.empty()
    states = p.empty_states(steps)
    before = j2d5pt.j2d5pt_kernel_launches()
    p.run_states(src, states, steps)
    assert j2d5pt.j2d5pt_kernel_launches() - before == 1 + launches  # the rings of all states in one
    p.set("algo", "onestep").run(src, one, steps)
    p.sync()
    assert torch.equal(p.view(states[steps - 1]), p.view(one))
    p.close()
