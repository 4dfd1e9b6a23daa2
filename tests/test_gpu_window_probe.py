"""Where a unit's window is chosen and given up: the first units of a band (whose
pipeline starts above the grid), rows that end a window early and late, units tall
enough for a second attempt, fields that are zero inside a hot ring, infinities
and NaNs.  Bit for bit against the one-step kernel."""
import numpy as np
import pytest

from paper_2306_03336_gb300 import j2d5pt

pytestmark = pytest.mark.gpu

W5 = np.array([0.5, 0.25, 0.04, 0.15, 0.06])
W9 = np.array([0.18, 0.03, 0.09, 0.12, 0.15, 0.11, 0.07, 0.17, 0.08])


def field(name, nx, ny):
    r = np.random.default_rng(6)
    u = 0.5 + 0.5 * r.random((ny + 2, nx + 2))
    if name == "hot_ring":
        u[1:-1, 1:-1] = 0.0
    elif name == "first_row":  # the first interior row fits no window
        u[1, 1:-1] *= 2.0 ** r.integers(-30, 30, size=nx)
    elif name == "fifth_row":  # the first row after the probed ones
        u[5, nx // 2] = 2.0 ** 30
    elif name == "last_row":
        u[ny, nx // 2] = -1.0
    elif name == "not_finite":
        u[ny // 3, nx // 2] = np.inf
        u[ny // 2, nx // 3] = -np.inf
        u[2 * ny // 3, nx - 1] = np.nan
    elif name == "not_finite_ring":
        u[0, nx // 2], u[ny // 2, 0], u[ny + 1, 1], u[ny // 3, nx + 1] = np.inf, np.nan, -np.inf, np.inf
    return u


def run(make, u, steps, algo, depth):
    plan = make().set("algo", algo).set("depth", depth)
    src, dst = plan.to_device(u), plan.empty()
    plan.run(src, dst, steps)
    plan.sync()
    got = plan.to_host(dst)
    plan.close()
    return got


@pytest.mark.parametrize("name", ["plain", "hot_ring", "first_row", "fifth_row", "last_row", "not_finite", "not_finite_ring"])
@pytest.mark.parametrize("nx,ny", [(130, 9), (187, 64), (61, 301)])
def test_probe_fields(name, nx, ny):
    u = field(name, nx, ny)

    def five():
        return j2d5pt.Plan(nx, ny, "f64", W5)

    def box():
        return j2d5pt.Plan.box9(nx, ny, "f64", W9)

    for make, depths in ((five, (2, 3, 4)), (box, (2,))):
        for steps in (4, 9):
            ref = run(make, u, steps, "onestep", 0)
            for depth in depths:
                got = run(make, u, steps, "stream", depth)
                assert np.array_equal(got, ref, equal_nan=True), (depth, steps)


def test_second_attempt_in_a_tall_unit():
    """52000 columns are more bands than warps run at once, so units are 268 rows tall:
    where their first rows fit no window, the attempt after 256 rows does."""
    import torch
    nx, ny, steps, depth = 52000, 2140, 4, 4
    plan = j2d5pt.Plan(nx, ny, "f64", W5)
    g = torch.Generator(device="cuda").manual_seed(7)
    src, ref, got = plan.empty(), plan.empty(), plan.empty()
    u = plan.view(src)
    u.copy_(0.5 + 0.5 * torch.rand(u.shape, generator=g, device="cuda", dtype=torch.float64))
    u[1::268] *= -1.0
    plan.set("algo", "onestep").run(src, ref, steps)
    plan.set("algo", "stream").set("depth", depth).run(src, got, steps)
    plan.sync()
    assert torch.equal(plan.view(got), plan.view(ref))
    plan.close()


@pytest.mark.parametrize("name", ["rise", "fall", "steep", "diagonal", "crossing"])
@pytest.mark.parametrize("nx,ny", [(130, 9), (187, 301), (61, 1203)])
def test_sloping_fields(name, nx, ny):
    """Fields whose exponents drift down a unit: into its window and out of it, with weights
    that leave eight binades and four."""
    y, x = np.arange(ny + 2)[:, None], np.arange(nx + 2)[None, :]
    u = {"rise": 2.0 ** (y / 30 + 0 * x), "fall": 2.0 ** (-y / 30 + 0 * x), "steep": 2.0 ** (y / 3 % 200 + 0 * x),
         "diagonal": 2.0 ** ((x + y) / 37 % 60), "crossing": 1 + 0.5 * np.sin(y / 20) * np.cos(x / 30)}[name]
    u = u * (1 + 2.0 ** -20 * np.random.default_rng(9).random(u.shape))
    narrow5 = np.array([0.55, 0.2, 0.0085, 0.13, 0.1115])
    narrow9 = np.array([0.25, 0.0085, 0.09, 0.12, 0.15, 0.11, 0.07, 0.1315, 0.07])
    for make, depths in ((lambda: j2d5pt.Plan(nx, ny, "f64", W5), (2, 3, 4)),
                         (lambda: j2d5pt.Plan(nx, ny, "f64", narrow5), (2, 4)),
                         (lambda: j2d5pt.Plan.box9(nx, ny, "f64", W9), (2,)),
                         (lambda: j2d5pt.Plan.box9(nx, ny, "f64", narrow9), (2,))):
        ref = run(make, u, 8, "onestep", 0)
        for depth in depths:
            assert np.array_equal(run(make, u, 8, "stream", depth), ref), depth
