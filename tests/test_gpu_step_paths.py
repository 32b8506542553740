"""Each path a step can take, at sizes that reach it: step graphs for more markers than the
one-kernel steps hold, against the same steps driven from the host; and the marker windows
of the sweeps at awkward shapes, which small plasmas do not use unless driven from the host."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2203_06513_gb300 import inputs as I
from paper_2203_06513_gb300 import pic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _markers_of_one_kernel():
    return 256 * torch.cuda.get_device_properties(0).multi_processor_count


FORMS = {
    "fp64": {},
    "fp64_explicit": dict(warm_start=1),
    "fp64_predicted": dict(warm_start=1, warm_field=1),
    "strang": dict(splitting=1),
    "strang_predicted": dict(splitting=1, warm_start=1, warm_field=1),
    "fp32_none": dict(precision=pic.PIC_FP32),
    "fp32_explicit": dict(precision=pic.PIC_FP32, warm_start=1),
    "fp32_predicted": dict(precision=pic.PIC_FP32, warm_start=1, warm_field=1),
    "fp32_strang": dict(precision=pic.PIC_FP32, splitting=1, warm_start=1),
    "fp32_float_lanes": dict(precision=pic.PIC_FP32, deposit=pic.PIC_ACC_FLOAT),
}


@pytest.mark.parametrize("form", FORMS)
def test_graph_steps_match_host_loops(form, monkeypatch):
    """Above the one-kernel limit, across marker sorts (one graph per marker copy).  The same
    iteration: the same sweep counts in double, and the tolerances of the comparison of
    small runs."""
    n = _markers_of_one_kernel() + 21099
    w = I.Workload("g", nx=96, degree=3, np=n, seed=23, vth=0.15, pump=0.25)
    cfg = pic.Config.from_workload(w, sort_every=2, **FORMS[form])
    double = cfg.precision == pic.PIC_FP64
    runs = []
    for no_graph in (False, True):
        if no_graph:
            monkeypatch.setenv("PIC_NO_GRAPH", "1")
        x, p = I.particles(w)
        g = pic.Pic(cfg, x, p, *I.fields(w))
        its = [g.step(1), g.step(6)]
        runs.append((g.state_numpy(), its, g.energy()))
        g.close()
    (a, ia, Ea), (b, ib, Eb) = runs
    if double:
        assert ia == ib
    else:   # float decisions near the noise floor may differ by a sweep a step (atomics order)
        for (a1, a2), (b1, b2) in zip(ia, ib):
            assert abs(a1 - b1) <= 14 and abs(a2 - b2) <= 7
    tol = 1e-12 if double else 1e-6
    d = np.abs(np.mod(a["x"] - b["x"] + 0.5 * w.L, w.L) - 0.5 * w.L)
    assert np.max(d) / w.L < tol
    for key in ("p", "ex", "ey", "ay"):
        assert np.max(np.abs(a[key] - b[key])) <= tol * np.max(np.abs(b[key])), key
    assert abs(Ea["total"] - Eb["total"]) < (1e-13 if double else 1e-10) * Eb["total"]


#       nx   k  markers   dt  vth  sort  z
SHAPES = [(33, 3, 2001, 0.05, 0.1, 0, True),
          (17, 2, 515, 0.05, 0.3, 2, False),
          (255, 5, 4099, 0.05, 0.15, 1, True),
          (8, 3, 33, 0.3, 0.5, 0, True),
          (9, 4, 1000, 0.5, 0.5, 1, False),
          (250, 3, 3000, 0.3, 0.8, 0, True),     # paths over several cells, unsorted
          (127, 5, 31, 0.1, 0.2, 0, False),
          (64, 4, 20011, 0.05, 0.1, 2, True)]


@pytest.mark.parametrize("shape,precision", [(s, pic.PIC_FP64) for s in SHAPES] +
                         [(s, pic.PIC_FP32) for s in SHAPES if s[2] >= 2000 and s[3] <= 0.05])
def test_windows_at_awkward_shapes(shape, precision, monkeypatch):
    """Host-driven steps, whose sweeps deposit through the windows, against the oracle, to the
    tolerances of the parity tests for a few steps."""
    monkeypatch.setenv("PIC_NO_GRAPH", "1")
    nx, k, n, dt, vth, sort, z = shape
    w = I.Workload("c", nx=nx, degree=k, np=n, dt=dt, vth=vth, pump=0.2, seed=nx + k)
    x, p = I.particles(w)
    ay, az, ey, ez = I.fields(w)
    if z:
        az = 0.05 * np.random.default_rng(k).normal(size=nx)
    x[: n // 4] = 3.5 * w.dx                       # a pile in one cell
    x[n // 4: n // 4 + 4] = [0.0, w.dx, np.nextafter(w.L, 0.0), 2 * w.dx]
    orc = O.Oracle(w.L, nx, k, w.weight, dt, w.tol, 200)
    s = O.initial_state(orc, x, p, ay, az, ey, ez)
    cfg = pic.Config.from_workload(w, precision=precision, sort_every=sort, max_iter=200, warm_start=1, warm_field=1)
    g = pic.Pic(cfg, x, p, ay, az, ey, ez)
    for _ in range(3):
        s = orc.step(s)
    g.step(3)
    st = g.state_numpy()
    tol_x, tol = (1e-11, 1e-10) if precision == pic.PIC_FP64 else (1e-5, 1e-4)
    d = np.mod(st["x"] - s.x + 0.5 * w.L, w.L) - 0.5 * w.L
    assert np.max(np.abs(d)) / w.L <= tol_x
    for key in ("p", "ex", "ey", "ez", "ay", "az"):
        ref = getattr(s, key)
        assert np.max(np.abs(st[key] - ref)) <= tol * max(np.max(np.abs(ref)), 1e-3), key
    if precision == pic.PIC_FP64:
        assert g.energy()["gauss"] < 1e-12
    g.close()
