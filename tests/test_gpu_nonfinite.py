"""Infinities and NaNs in the ring and beside it.  Forward, ring cells are held whatever
their neighbours are.  Adjoint, a cell takes nothing from the ring (a NaN there stays
where it is), and a ring cell adds its one interior neighbour.  The infinities and
NaNs of a run are those of the plain sums."""
import numpy as np
import pytest

from paper_2306_03336_gb300 import j2d5pt, synth

pytestmark = pytest.mark.gpu

WEIGHTS = np.array([0.5, 0.25, 0.04, 0.15, 0.06])  # x - 1, x + 1, y - 1, centre, y + 1


def forward(u, steps):
    W, E, S, C, N = WEIGHTS
    for _ in range(steps):
        n = u.copy()
        n[1:-1, 1:-1] = W * u[1:-1, :-2] + E * u[1:-1, 2:] + S * u[:-2, 1:-1] + C * u[1:-1, 1:-1] + N * u[2:, 1:-1]
        u = n
    return u


def backward(lam, steps):
    lam = lam.copy()
    for _ in range(steps):
        inner, lam = lam[1:-1, 1:-1], lam.copy()
        lam[1:-1, 1:-1] = 0.0
        ny, nx = inner.shape
        for w, (dy, dx) in zip(WEIGHTS, ((0, -1), (0, 1), (-1, 0), (0, 0), (1, 0))):
            lam[1 + dy:1 + dy + ny, 1 + dx:1 + dx + nx] += w * inner
    return lam


def field(where, nx, ny):
    u = 0.5 + 0.5 * np.random.default_rng(8).random((ny + 2, nx + 2))
    if where == "beside":
        u[1, 1], u[ny, nx], u[ny // 2 + 1, 1], u[1, nx // 2 + 1] = np.inf, -np.inf, np.nan, np.inf
    else:
        u[0, nx // 2], u[ny // 2, 0], u[ny + 1, nx // 3], u[ny // 3, nx + 1] = np.inf, np.nan, -np.inf, np.inf
        u[0, 0], u[ny + 1, nx + 1] = np.nan, np.inf
    return u


def compare(got, ref, dt, steps):
    finite = np.isfinite(ref)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.array_equal(got[np.isinf(ref)], ref[np.isinf(ref)])
    # positive terms: five roundings a step, in FP32 a sixth for the weights
    bound = 5 * 2.0 ** -52 if dt == "f64" else 6 * 2.0 ** -23
    assert np.all(np.abs(got[finite] - ref[finite]) <= bound * steps * ref[finite])


def prepared(where, nx, ny, dt, algo):
    u = field(where, nx, ny)
    if dt == "f32":
        u = u.astype(np.float32)
    plan = j2d5pt.Plan(nx, ny, dt, WEIGHTS).set("algo", algo)
    return plan, plan.to_device(u), plan.empty(), u.astype(np.float64)


SIZES = [(5, 3), (62, 40), (63, 41), (126, 30), (187, 64)]


@pytest.mark.parametrize("where", ["ring", "beside"])
@pytest.mark.parametrize("dt", ["f64", "f32"])
@pytest.mark.parametrize("algo", ["onestep", "stream"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_forward(nx, ny, algo, dt, where):
    plan, src, dst, u = prepared(where, nx, ny, dt, algo)
    for steps in (1, 5):
        plan.run(src, dst, steps)
        plan.sync()
        with np.errstate(invalid="ignore"):
            compare(plan.to_host(dst), forward(u, steps), dt, steps)
    plan.close()


@pytest.mark.parametrize("where", ["ring", "beside"])
@pytest.mark.parametrize("nx,ny,dt,algo", [(x, y, dt, "onestep") for x, y in SIZES for dt in ("f64", "f32")] +
                         [(187, 64, "f64", "tiles"), (2304, 1700, "f64", "auto")])
def test_adjoint(nx, ny, dt, algo, where):
    plan, src, dst, lam = prepared(where, nx, ny, dt, algo)
    for steps in (1, 5):
        plan.run_adjoint(src, dst, steps)
        plan.sync()
        with np.errstate(invalid="ignore"):
            compare(plan.to_host(dst), backward(lam, steps), dt, steps)
    plan.close()


@pytest.mark.parametrize("where", ["ring", "beside"])
@pytest.mark.parametrize("dt", ["f64", "f32"])
def test_fused_adjoint_step(dt, where):
    import torch
    nx, ny = 187, 64
    plan, src, dst, lam = prepared(where, nx, ny, dt, "auto")
    u = plan.to_device(synth.field(nx, ny, 61).astype(np.float32 if dt == "f32" else np.float64))
    plan.adjoint_step_wgrad(u, src, dst, torch.zeros(5, dtype=torch.float64, device="cuda"))
    plan.sync()
    with np.errstate(invalid="ignore"):
        compare(plan.to_host(dst), backward(lam, 1), dt, 1)
    plan.close()
