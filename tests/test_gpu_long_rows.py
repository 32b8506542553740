"""Solves whose inverse rows are long (large dt/dx): their nodes are formed in a pass before
the solve.  The one-kernel steps and the host loops against the oracle (both sides solve the
same fixed point to 1e-13 and differ in rounding order, as in the parity tests), graphs
and ensembles against the host loops."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2203_06513_gb300 import inputs as I
from paper_2203_06513_gb300 import pic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

#       nx   k  dt/dx: the row is the whole circle, half of it, a pass without need for it next to it
SHAPES = [(513, 5, 64.0), (1031, 4, 8.0), (640, 3, 16.0), (255, 2, 2.0)]


def _case(nx, k, r, n):
    L = nx / r * 0.2
    x = (np.arange(n) + 0.5) / n * L
    rng = np.random.default_rng(nx)
    p = 0.1 * rng.normal(size=n)
    q = 2 * np.pi / L * np.arange(nx) * L / nx
    ay, ey = 0.1 * np.cos(q), 0.05 * np.sin(q)
    az, ez = 0.05 * np.sin(2 * q), 0.02 * np.cos(q)
    return L, x, p, ay, az, ey, ez


def _compare(st, ref, L, tol):
    d = np.mod(st["x"] - ref["x"] + 0.5 * L, L) - 0.5 * L
    assert np.max(np.abs(d)) / L <= 0.1 * tol
    for key in ("p", "ex", "ey", "ez", "ay", "az"):
        assert np.max(np.abs(st[key] - ref[key])) <= tol * max(np.max(np.abs(ref[key])), 1e-3), key


@pytest.mark.parametrize("no_graph", [False, True])
@pytest.mark.parametrize("nx,k,r", SHAPES)
def test_long_rows_vs_oracle(nx, k, r, no_graph, monkeypatch):
    if no_graph:
        monkeypatch.setenv("PIC_NO_GRAPH", "1")
    n, dt, tol = 2003, 0.2, 1e-13
    L, x, p, ay, az, ey, ez = _case(nx, k, r, n)
    orc = O.Oracle(L, nx, k, L / n, dt, tol, 200)
    s = O.initial_state(orc, x, p, ay, az, ey, ez)
    g = pic.Pic(pic.Config(L, nx, k, n, L / n, dt, tol=tol, max_iter=200, warm_start=1, warm_field=1), x, p, ay, az, ey, ez)
    for _ in range(2):
        s = orc.step(s)
    g.step(2)
    _compare(g.state_numpy(), {q: getattr(s, q) for q in ("x", "p", "ex", "ey", "ez", "ay", "az")}, L, 1e-10)
    g.close()


@pytest.mark.parametrize("precision", [pic.PIC_FP64, pic.PIC_FP32])
@pytest.mark.parametrize("nx,k,r", SHAPES)
def test_long_rows_graph_and_ensemble_vs_host_loops(nx, k, r, precision, monkeypatch):
    """The host-driven steps of the same kernels: rounding order apart the same state (1e-11
    of a field in double; the float form's decisions near its noise may differ by a sweep)."""
    n, dt = 40003, 0.2
    tol = 1e-13 if precision == pic.PIC_FP64 else 1e-9
    L, *f = _case(nx, k, r, n)
    cfg = pic.Config(L, nx, k, n, L / n, dt, tol=tol, max_iter=200, precision=precision, warm_start=1, warm_field=1)
    x, p, ay, az, ey, ez = f
    g = pic.Pic(cfg, *f)
    g.step(4)
    got = g.state_numpy()
    g.close()
    e = pic.Ensemble([cfg] * 3, [(x, p, ay, az, ey, ez)] * 3)
    e.step(4)
    runs = [e.run(q).state_numpy() for q in range(3)]
    e.close()
    monkeypatch.setenv("PIC_NO_GRAPH", "1")
    h = pic.Pic(cfg, *f)
    h.step(4)
    ref = h.state_numpy()
    h.close()
    for st in [got] + runs:
        _compare(st, ref, L, 1e-11 if precision == pic.PIC_FP64 else 1e-4)
