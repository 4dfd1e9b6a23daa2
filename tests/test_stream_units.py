"""What the stream schedule's warps store (host arithmetic, no device): the rows of a
band each once, runs cut into whole numbers of units, units as tall as their minimum, and
enough of them to fill the device where the runs alone do not."""
import numpy as np
import pytest

from paper_2306_03336_gb300 import j2d5pt


def cases():
    yield from [(16384, 16384, "f64", 2, 3040), (4096, 4096, "f64", 2, 3040), (2048, 1536, "f32", 6, 2400), (512, 512, "f32", 6, 2400),
                (1, 1, "f64", 4, 1), (3, 700, "f32", 4, 4000), (700, 3, "f64", 6, 100), (52000, 2140, "f64", 4, 1824)]
    rng = np.random.Generator(np.random.PCG64(2306034901))
    for _ in range(200):
        dt = str(rng.choice(["f64", "f32"]))
        depth = int(rng.choice([2, 3, 4, 6] if dt == "f64" else [4, 6, 8, 10, 12]))
        yield (int(rng.integers(1, 20000)), int(rng.integers(1, 20000)), dt, depth, int(rng.integers(1, 5000)))


def test_units_store_every_row_once():
    for nx, ny, dt, depth, warps in cases():
        q = j2d5pt.j2d5pt_stream_geometry(nx, ny, dt, depth, warps)
        rows, units = j2d5pt.j2d5pt_stream_units(nx, ny, dt, depth, warps)
        stored = np.zeros(ny + 2, dtype=np.int64)
        for u in range(units):
            lo, hi = 1 + u * rows, min(1 + (u + 1) * rows, ny + 1)
            assert lo <= ny
            assert (lo - 1) // q["H"] == (hi - 2) // q["H"]  # in one run
            stored[lo:hi] += 1
        assert (stored[1:ny + 1] == 1).all(), (ny, rows, units)
        assert q["H"] % rows == 0
        least = 8 if dt == "f64" else 7 * depth // 2
        assert rows >= min(least, ny), (ny, rows)
        if rows < q["H"]:  # shared runs: no more warps than the device holds, unless a unit is at its minimum
            assert q["bands"] * units <= warps or rows == least or q["bands"] > warps, (nx, ny, dt, depth, warps)


def test_units_errors():
    for bad in [(0, 5, "f64", 2, 10, 5), (5, 5, "f64", 5, 10, 5), (5, 5, "f64", 2, 0, 5), (5, 5, "f64", 6, 10, 9)]:
        with pytest.raises(j2d5pt.J2DError) as e:
            j2d5pt.j2d5pt_stream_units(*bad[:5], shape=bad[5])
        assert e.value.status == j2d5pt.J2D_ERR_ARG
