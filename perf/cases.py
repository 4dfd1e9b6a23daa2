"""Cases that time this library the way its users call it.

A case is a dict of plain values:

- "op": "run" (Plan.run), "batch" (Plan.run_batched, replayed as a CUDA
  graph), "adjoint" (Plan.run_adjoint), "grad" (forward and backward through
  autograd.J2D5PT) or "host" (Plan.run_host, pinned host arrays in and out);
- "shape": 5 (j2d5pt) or 9 (the 3x3 box); "dtype": "f64" or "f32";
- "nx", "ny", "steps" (a batch: "count" grids with sides "lo".."hi", drawn
  from the seed "sizes");
- "field": "uniform", values in [0, 1), the repository's own inputs, or
  "signed", values in [-1, 1), as gradients and centred fields have them.

Every plan keeps its default options (the library's own choice of kernel),
except that a batch is replayed as a CUDA graph.  The sizes are those of the
library's workloads (512^2, 2048x1536, 16384^2, 8592x8328, 4096^2, 256 grids
with sides 64..1024), fewer steps where a thousand would take seconds, and odd
sizes between them.
"""
import math

import numpy as np
import torch

from paper_2306_03336_gb300 import autograd, j2d5pt

CHECKPOINT = 50  # steps between the checkpoints of a gradient run


def listed():
    return [
        # the smallest call a program makes: a check or a step of a control loop, latency only
        _case("small_f64", nx=200, ny=120, steps=12),
        # a small grid and a short run
        _case("f64_512", nx=512, ny=512, steps=16),
        # a grid that fits on the chip, relaxed for a thousand steps
        _case("onchip_f64", nx=2048, ny=1536, steps=1000),
        # a grid beyond the chip's shared memory with odd sides
        _case("odd_f64", nx=3001, ny=4099, steps=100),
        # the largest grid in double precision
        _case("large_f64", nx=16384, ny=16384, steps=48),
        # the same grid in single precision
        _case("large_f32", nx=16384, ny=16384, steps=200, dtype="f32"),
        # single precision on the chip, odd sides
        _case("onchip_f32", nx=1531, ny=2047, steps=500, dtype="f32"),
        # the nine-point stencil in both precisions, a square grid and a ragged one
        _case("box_f64", nx=4096, ny=4096, steps=64, shape=9),
        _case("box_f32", nx=8592, ny=8328, steps=96, shape=9, dtype="f32"),
        # many independent grids of uneven sizes
        {"name": "batch_f64", "op": "batch", "shape": 5, "dtype": "f64", "count": 256, "lo": 64, "hi": 1024,
         "sizes": 3, "steps": 200, "field": "uniform"},
        # the gradient of a loss with respect to the initial field alone (signed, as gradients are)
        _case("adjoint_f64", op="adjoint", nx=4096, ny=4096, steps=100, field="signed"),
        # a training step: forward, then the gradient in the field and the weights
        _case("grad_f64", op="grad", nx=4096, ny=4096, steps=100),
    ]


def _case(name, op="run", nx=0, ny=0, steps=1, dtype="f64", shape=5, field="uniform"):
    return {"name": name, "op": op, "shape": shape, "dtype": dtype, "nx": nx, "ny": ny, "steps": steps,
            "field": field}


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op, shape, dtype = rng.choice([
        ("run", 5, "f64"), ("run", 5, "f64"), ("run", 5, "f32"), ("run", 5, "f32"), ("run", 9, "f64"),
        ("run", 9, "f32"), ("batch", 5, "f64"), ("batch", 5, "f32"), ("adjoint", 5, "f64"), ("grad", 5, "f64"),
        ("host", 5, "f64")])
    field = rng.choice(["uniform", "uniform", "uniform", "signed"])
    if op == "batch":
        hi = log_int(128, 1024)
        count = log_int(8, 256)
        cells = count * (0.5 * (64 + hi)) ** 2
        steps = max(1, min(log_int(10, 200), int(8e9 / cells)))
        return {"op": op, "shape": shape, "dtype": dtype, "count": count, "lo": 64, "hi": hi,
                "sizes": rng.randrange(1 << 20), "steps": steps, "field": field}
    top = 4096 if op in ("grad", "host") else 8192 if op == "adjoint" else 16384
    nx, ny = log_int(64, top), log_int(64, top)
    most = {"grad": 1e9, "adjoint": 3e9, "host": 2e9}.get(op, 4e9 if shape == 9 else 8e9)
    steps = max(1, min(log_int(1, 1000), int(most / (nx * ny))))
    return {"op": op, "shape": shape, "dtype": dtype, "nx": nx, "ny": ny, "steps": steps, "field": field}


def _sizes(case):
    """Interior (nx, ny) of every grid of the case."""
    if case["op"] != "batch":
        return [(case["nx"], case["ny"])]
    r = np.random.default_rng(case["sizes"])
    side = r.integers(case["lo"], case["hi"] + 1, size=(case["count"], 2))
    return [(int(a), int(b)) for a, b in side]


def _weights(case, seed, count):
    """Normalised positive weights, one set per grid."""
    w = np.random.default_rng([seed, 2]).random((count, case["shape"]))
    return w / w.sum(axis=1, keepdims=True)


def _torch_dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _fields(case, seed, sizes):
    """A (ny+2, nx+2) field per grid, ring included, on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for nx, ny in sizes:
        t = torch.rand((ny + 2, nx + 2), generator=g, device="cuda", dtype=_torch_dtype(case))
        out.append(t if case["field"] == "uniform" else t.mul_(2.0).sub_(1.0))
    return out


def prepare(case, seed):
    sizes = _sizes(case)
    w = _weights(case, seed, len(sizes))
    fields = _fields(case, seed, sizes)
    state = {"op": case["op"], "steps": case["steps"]}
    if case["op"] == "grad":
        g = torch.Generator(device="cuda").manual_seed(seed + 1)
        state["operator"] = autograd.J2D5PT(case["nx"], case["ny"], case["dtype"], checkpoint=CHECKPOINT)
        state["u0"] = fields[0].requires_grad_(True)
        state["w"] = torch.from_numpy(w[0]).cuda().requires_grad_(True)
        # dL/du_T of the loss sum(c * u_T)
        state["c"] = torch.rand(fields[0].shape, generator=g, device="cuda", dtype=fields[0].dtype)
        return state
    if case["op"] == "batch":
        plan = j2d5pt.Plan.batch(sizes, case["dtype"], w)
        plan.set("graph", 1)
    elif case["shape"] == 9:
        plan = j2d5pt.Plan.box9(case["nx"], case["ny"], case["dtype"], w[0])
    else:
        plan = j2d5pt.Plan(case["nx"], case["ny"], case["dtype"], w[0])
    state["plan"] = plan
    if case["op"] == "host":
        state["in"] = fields[0].cpu().pin_memory().numpy()
        state["out"] = torch.empty(fields[0].shape, dtype=fields[0].dtype).pin_memory().numpy()
        return state
    state["src"] = [plan.empty(i) for i in range(len(sizes))]
    state["dst"] = [plan.empty(i) for i in range(len(sizes))]
    for i, f in enumerate(fields):
        plan.view(state["src"][i], i).copy_(f)
    return state


def run(state):
    op, steps = state["op"], state["steps"]
    if op == "grad":
        u0, w = state["u0"], state["w"]
        out = state["operator"](u0, w, steps)
        du0, dw = torch.autograd.grad(out, (u0, w), state["c"])
        return {"out": out.detach(), "du0": du0, "dw": dw}
    plan = state["plan"]
    if op == "host":
        return {"out": plan.run_host(state["in"], steps, out=state["out"])}
    src, dst = state["src"], state["dst"]
    if op == "batch":
        plan.run_batched(src, dst, steps)
        # the grids one after another, as one array
        return {"out": torch.cat([plan.view(t, i).reshape(-1) for i, t in enumerate(dst)])}
    if op == "adjoint":
        plan.run_adjoint(src[0], dst[0], steps)
    else:
        plan.run(src[0], dst[0], steps)
    return {"out": plan.view(dst[0])}


def work(case):
    """Each input read once and each output written once; 9 flops per five-point
    cell update (17 for the box), 10 more per cell and step for the weight gradient."""
    elem = 8 if case["dtype"] == "f64" else 4
    if case["op"] == "batch":
        mean = 0.5 * (case["lo"] + case["hi"])
        cells, all_cells = case["count"] * mean ** 2, case["count"] * (mean + 2) ** 2
    else:
        cells, all_cells = case["nx"] * case["ny"], (case["nx"] + 2) * (case["ny"] + 2)
    per_step = 17 if case["shape"] == 9 else 9
    arrays = 2
    if case["op"] == "grad":
        per_step, arrays = 9 + 9 + 10, 4  # u0 and dL/du_T in, u_T and dL/du_0 out
    return {"bytes": arrays * elem * all_cells, "flops": per_step * cells * case["steps"]}


# ---- the same results in 64 bits, plain torch ------------------------------------


def _neighbours(shape):
    """Offsets (dy, dx) in the order of the weights."""
    if shape == 9:
        return [(dy, dx) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
    return [(0, -1), (0, 1), (-1, 0), (0, 0), (1, 0)]  # W, E, S, C, N


def _shifted(u, dy, dx):
    ny, nx = u.shape[0] - 2, u.shape[1] - 2
    return u[1 + dy:1 + dy + ny, 1 + dx:1 + dx + nx]


def _forward(u, w, shape, steps, keep=None):
    u = u.clone()
    for _ in range(steps):
        if keep is not None:
            keep.append(u.clone())
        new = None
        for wd, (dy, dx) in zip(w, _neighbours(shape)):
            term = _shifted(u, dy, dx) * wd
            new = term if new is None else new.add_(term)
        u[1:-1, 1:-1] = new
    return u


def _backward(lam, w, steps, states=None):
    """lam_0 and, with the forward's states, the weight gradient."""
    lam = lam.clone()
    dw = torch.zeros(5, dtype=torch.float64, device=lam.device)
    for t in reversed(range(steps)):
        inner = lam[1:-1, 1:-1].clone()
        if states is not None:
            for d, (dy, dx) in enumerate(_neighbours(5)):
                dw[d] += (inner * _shifted(states[t], dy, dx)).sum()
        lam[1:-1, 1:-1] = 0.0
        for wd, (dy, dx) in zip(w, _neighbours(5)):
            _shifted(lam, dy, dx).add_(inner, alpha=wd)
    return lam, dw


def exact(case, seed):
    sizes = _sizes(case)
    w = _weights(case, seed, len(sizes))
    if case["dtype"] == "f32":
        w = w.astype(np.float32).astype(np.float64)  # a single-precision plan holds its weights in FP32
    fields = [f.double() for f in _fields(case, seed, sizes)]
    steps, shape = case["steps"], case["shape"]
    wl = [[float(v) for v in row] for row in w]
    if case["op"] == "batch":
        outs = [_forward(f, wi, shape, steps) for f, wi in zip(fields, wl)]
        return {"out": torch.cat([o.reshape(-1) for o in outs])}
    if case["op"] == "adjoint":
        return {"out": _backward(fields[0], wl[0], steps)[0]}
    if case["op"] == "grad":
        g = torch.Generator(device="cuda").manual_seed(seed + 1)
        c = torch.rand(fields[0].shape, generator=g, device="cuda", dtype=_torch_dtype(case)).double()
        states = []
        out = _forward(fields[0], wl[0], shape, steps, keep=states)
        du0, dw = _backward(c, wl[0], steps, states)
        return {"out": out, "du0": du0, "dw": dw}
    return {"out": _forward(fields[0], wl[0], shape, steps)}
