"""The tuning cache's key tells plans apart whose weights the integer path treats
differently (a window, positive without one, chains only), and holds nothing of the weights
beyond that."""
import numpy as np
import pytest

from paper_2306_03336_gb300 import j2d5pt, synth

pytestmark = pytest.mark.gpu

NX, NY, STEPS = 200, 120, 8


def tuned(w, dt="f64", path=1):
    plan = j2d5pt.Plan(NX, NY, dt, np.array(w)).set("int_path", path)
    u = synth.field(NX, NY, 81)
    src, dst = plan.to_device(u.astype(np.float32) if dt == "f32" else u), plan.empty()
    plan.autotune(src, dst, STEPS)
    plan.close()


def test_keys(tmp_path, monkeypatch):
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("J2D_TUNE_CACHE", str(cache))

    def keys():
        return [line.split()[0] for line in cache.read_text().splitlines()]

    tuned([0.5, 0.25, 0.04, 0.15, 0.06])
    tuned([0.2] * 5)  # another window: the same key, nothing tuned again
    assert len(keys()) == 1
    tuned([0.55, 0.2, 0.0005, 0.1395, 0.11])
    tuned([0.25, 0.25, 0.25, 0.0, 0.25])
    tuned([0.3, 0.3, -0.1, 0.25, 0.25])
    assert len(keys()) == 3 and len(set(keys())) == 3
    tuned([0.5, 0.25, 0.04, 0.15, 0.06], dt="f32")
    tuned([0.25, 0.25, 0.25, 0.0, 0.25], dt="f32")
    assert len(keys()) == 4
