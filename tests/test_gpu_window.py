"""FP64 stream sweeps in windowed fixed point against the one-step kernel, bit
for bit: values at and beyond the window's two ends (inside the grid, in the
ring rows and columns, at the edges of runs), fields no window holds, fields whose
window moves down the rows, weights at the limits of the fixed-point form (the
widest spread it takes, one more, a zero, a negative, significands of all ones)."""
import numpy as np
import pytest

from paper_2306_03336_gb300 import j2d5pt, synth

pytestmark = pytest.mark.gpu

ONES = float(np.nextafter(1.0, 0.0))
WEIGHTS = {
    "equal": [0.2] * 5,
    "spread4": [0.5, 0.25, 0.04, 0.15, 0.06],
    "spread5": [0.55, 0.2, 0.0175, 0.13, 0.1],
    "spread7": [0.55, 0.2, 0.0043, 0.13, 0.11],
    "spread8": [0.55, 0.2, 0.0021, 0.13, 0.11],
    "spread9": [0.55, 0.2, 0.0011, 0.13, 0.11],
    "all_large": [0.24, 0.24, 0.24, 0.24, 0.0012],
    "all_ones": [ONES / 4, ONES / 8, ONES / 4, ONES / 4, ONES / 8],
    "zero": [0.25, 0.25, 0.0, 0.25, 0.25],
    "negative": [0.3, 0.3, -0.1, 0.25, 0.25],
    "large": [30.0, 20.0, 10.0, 25.0, 15.0],
}


def field(name, nx, ny):
    r = np.random.default_rng(5)
    u = 0.5 + 0.5 * r.random((ny + 2, nx + 2))
    if name == "uniform":
        return r.random((ny + 2, nx + 2))
    if name == "spikes":  # single cells at both ends of the window and beyond it
        for v in [2.0 ** -6, 2.0 ** -7, 2.0 ** -7 * ONES, 2.0 ** -8, 1.0, 2.0, 2.0 * ONES, 4.0, 0.0, -1.0, 5e-324]:
            u[r.integers(0, ny + 2), r.integers(0, nx + 2)] = v
    elif name == "ring":  # ring values outside the window
        for edge in (u[0], u[-1], u[:, 0], u[:, -1]):
            edge[:] = r.choice([0.0, 1e-3, 0.7, 1e3, -2.0], size=edge.shape)
    elif name == "zero_ring":
        u[0], u[-1], u[:, 0], u[:, -1] = 0.0, 0.0, 0.0, 0.0
    elif name == "ramp":  # a window of its own every few rows
        u *= 2.0 ** (np.arange(ny + 2)[:, None] // 7 % 40 - 20)
    elif name == "wide":
        u *= 2.0 ** r.integers(-40, 40, size=u.shape)
    elif name == "tiny":  # below every window
        u *= 2.0 ** -1019
    elif name == "huge":
        u *= 2.0 ** 1000
    elif name == "short":  # rounding ties
        u = np.floor(u * 2 ** 12) / 2 ** 12
    return u


def run(u, w, nx, ny, steps, algo, depth):
    plan = j2d5pt.Plan(nx, ny, "f64", w).set("algo", algo).set("depth", depth)
    src, dst = plan.to_device(u), plan.empty()
    plan.run(src, dst, steps)
    plan.sync()
    got = plan.to_host(dst)
    plan.close()
    return got


@pytest.mark.parametrize("fname", ["uniform", "spikes", "ring", "zero_ring", "ramp", "wide", "tiny", "huge", "short"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 2), (61, 70), (124, 129), (187, 301)])
def test_window_fields(fname, nx, ny):
    u = field(fname, nx, ny)
    w = np.array(WEIGHTS["spread4"])
    for depth, steps in ((2, 5), (3, 7), (4, 8)):
        ref = run(u, w, nx, ny, steps, "onestep", 0)
        got = run(u, w, nx, ny, steps, "stream", depth)
        assert np.array_equal(got, ref), "k=%d: %d cells differ" % (depth, np.count_nonzero(got != ref))


@pytest.mark.parametrize("wname", sorted(WEIGHTS))
def test_window_weights(wname):
    nx, ny = 130, 203
    w = np.array(WEIGHTS[wname])
    for fname in ("spikes", "short"):
        u = field(fname, nx, ny)
        for depth, steps in ((2, 4), (3, 3)):
            ref = run(u, w, nx, ny, steps, "onestep", 0)
            got = run(u, w, nx, ny, steps, "stream", depth)
            assert np.array_equal(got, ref), "%s k=%d: %d cells differ" % (fname, depth, np.count_nonzero(got != ref))


@pytest.mark.parametrize("fname", ["uniform", "spikes", "ramp", "wide", "tiny", "short"])
@pytest.mark.parametrize("nx,ny", [(130, 12), (131, 9), (323, 70)])
def test_window_adjoint_items(fname, nx, ny):
    """Windowed items of the one-step adjoint, alone and with the weight gradient
    fused, against the tiles (no window)."""
    import torch
    for wname in ("spread4", "spread5", "spread9"):
        lam = field(fname, nx, ny)
        plan = j2d5pt.Plan(nx, ny, "f64", np.array(WEIGHTS[wname]))
        src, got, ref = plan.to_device(lam), plan.empty(), plan.empty()
        for steps in (1, 4):
            plan.set("algo", "tiles").set("depth", 2).run_adjoint(src, ref, steps)
            plan.set("algo", "onestep").run_adjoint(src, got, steps)
            plan.sync()
            assert np.array_equal(plan.to_host(got), plan.to_host(ref)), (wname, steps)
        u = plan.to_device(synth.field(nx, ny, 31))
        dw, dw2 = (torch.zeros(5, dtype=torch.float64, device="cuda") for _ in range(2))
        plan.set("algo", "tiles").run_adjoint(src, ref, 1)
        plan.adjoint_step_wgrad(u, src, got, dw)
        plan.weight_grad(u, src, dw2)
        plan.sync()
        assert np.array_equal(plan.to_host(got), plan.to_host(ref)), wname
        # two fixed summation orders of the same nx * ny products
        a, b = dw.cpu().numpy(), dw2.cpu().numpy()
        bound = 2.0 ** -52 * nx * ny * np.abs(lam).max() * 1.0
        assert np.all(np.abs(a - b) <= bound * nx * ny), wname
        plan.close()


@pytest.mark.parametrize("fname", ["uniform", "spikes", "ring", "ramp", "short"])
def test_window_states(fname):
    """State-keeping stream runs: every state against chained one-step runs."""
    nx, ny, steps = 187, 301, 7
    u = field(fname, nx, ny)
    for depth in (2, 3, 4):
        plan = j2d5pt.Plan(nx, ny, "f64", np.array(WEIGHTS["spread4"]))
        src = plan.to_device(u)
        states = plan.empty_states(steps)
        plan.set("algo", "stream").set("depth", depth).run_states(src, states, steps)
        plan.sync()
        plan.set("algo", "onestep")
        cur = src
        for t in range(steps):
            nxt = plan.empty()
            plan.run(cur, nxt, 1)
            plan.sync()
            assert np.array_equal(plan.to_host(states[t]), plan.to_host(nxt)), (depth, t)
            cur = nxt
        plan.close()


BOX_WEIGHTS = {
    "even": [1 / 9] * 9,
    "spread3": [0.18, 0.03, 0.09, 0.12, 0.15, 0.11, 0.07, 0.17, 0.08],
    "spread5": [0.25, 0.008, 0.09, 0.12, 0.15, 0.11, 0.07, 0.132, 0.07],
    "spread7": [0.25, 0.0018, 0.09, 0.12, 0.15, 0.11, 0.07, 0.138, 0.07],
    "zero": [0.125, 0.125, 0.125, 0.125, 0.0, 0.125, 0.125, 0.125, 0.125],
    "negative": [0.2, 0.1, -0.05, 0.15, 0.2, 0.1, 0.1, 0.1, 0.1],
}


@pytest.mark.parametrize("fname", ["uniform", "spikes", "ring", "zero_ring", "ramp", "wide", "tiny", "huge", "short"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 2), (61, 70), (124, 129), (187, 301)])
def test_window_box_fields(fname, nx, ny):
    u = field(fname, nx, ny)
    w = np.array(BOX_WEIGHTS["spread3"])
    for steps in (1, 4, 5):
        ref = run(u, w, nx, ny, steps, "onestep", 0)
        got = run(u, w, nx, ny, steps, "stream", 2)
        assert np.array_equal(got, ref), "%d steps: %d cells differ" % (steps, np.count_nonzero(got != ref))


@pytest.mark.parametrize("wname", sorted(BOX_WEIGHTS))
def test_window_box_weights(wname):
    nx, ny = 130, 203
    w = np.array(BOX_WEIGHTS[wname])
    for fname in ("spikes", "short"):
        u = field(fname, nx, ny)
        ref = run(u, w, nx, ny, 4, "onestep", 0)
        got = run(u, w, nx, ny, 4, "stream", 2)
        assert np.array_equal(got, ref), "%s: %d cells differ" % (fname, np.count_nonzero(got != ref))
