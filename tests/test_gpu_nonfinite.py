"""Positions that are not finite: every call ends at once and says so, in both forms and
on each path a step can take.  A marker whose position came in as NaN or infinity has no
end point; the steps return PIC_ERR_NUMERIC, and a deposit of given displacements returns
its contribution as NaN in the nodes of one cell."""
import ctypes

import numpy as np
import pytest

from paper_2203_06513_gb300 import inputs as I
from paper_2203_06513_gb300 import pic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BAD = [np.nan, np.inf, -np.inf]
FORMS = [pic.PIC_FP64, pic.PIC_FP32]


def _inputs(n, k, bad, nx=33):
    w = I.Workload("f", nx=nx, degree=k, np=n, dt=0.05, vth=0.1, pump=0.2, seed=n + k)
    x, p = I.particles(w)
    ay, az, ey, ez = I.fields(w)
    x[n // 2] = bad
    return w, x, p, ay, az, ey, ez


@pytest.mark.parametrize("precision", FORMS)
@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("n,warm,field,no_graph", [(2003, 0, 0, False), (2003, 1, 1, False), (2003, 0, 0, True),
                                                   (2003, 1, 0, True), (2003, 1, 1, True), (2003, 2, 0, True),
                                                   (40001, 1, 1, False), (1, 0, 0, False), (1, 0, 0, True)])
def test_steps_report_positions_that_are_not_finite(precision, bad, n, warm, field, no_graph, monkeypatch):
    if no_graph:
        monkeypatch.setenv("PIC_NO_GRAPH", "1")
    w, x, p, ay, az, ey, ez = _inputs(n, 3, bad)
    g = pic.Pic(pic.Config.from_workload(w, precision=precision, warm_start=warm, warm_field=field, sort_every=1),
                x, p, ay, az, ey, ez)
    if warm == pic.PIC_WARM_MLP:
        net = pic.Mlp(np.r_[np.zeros(6), np.ones(8)])
        net.attach(g)
    with pytest.raises(pic.PicError) as e:
        g.step(2)
    assert e.value.code == pic.PIC_ERR_NUMERIC
    g.close()


@pytest.mark.parametrize("precision", FORMS)
@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("field", [0, 1])
def test_a_bad_run_of_an_ensemble_stops_alone(precision, bad, field):
    kw = dict(precision=precision, warm_start=1, warm_field=field)
    w, x, p, *f = _inputs(3001, 3, 0.25)
    cfg = pic.Config.from_workload(w, **kw)
    xb = x.copy()
    xb[7] = bad
    e = pic.Ensemble([cfg, cfg, cfg], [(x, p, *f), (xb, p, *f), (x, p, *f)])
    sweeps, status = e.step(3, check=False)
    assert list(status) == [0, pic.PIC_ERR_NUMERIC, 0]
    assert np.all(sweeps[[0, 2]] >= 3)
    for r in (0, 2):
        assert np.all(np.isfinite(e.run(r).state_numpy()["ex"]))
    e.close()


@pytest.mark.parametrize("precision", FORMS)
@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("k", [2, 5])
def test_current_of_a_position_that_is_not_finite(precision, bad, k):
    w, x, p, ay, az, ey, ez = _inputs(500, k, bad)
    g = pic.Pic(pic.Config.from_workload(w, precision=precision), x, p, ay, az, ey, ez)
    d = torch.full((w.np,), 0.3 * w.dx, dtype=torch.float64, device="cuda")
    out = torch.zeros(w.nx, dtype=torch.float64, device="cuda")
    g.deposit(pic.PIC_DEP_CURRENT, d, out)
    lost = np.count_nonzero(~np.isfinite(out.cpu().numpy()))
    assert 1 <= lost <= k
    g.close()


@pytest.mark.parametrize("precision", FORMS)
@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("k", [2, 5])
def test_charge_of_a_position_that_is_not_finite(precision, bad, k):
    """Its nodes are NaN, and with them the field of the discrete Poisson equation."""
    w, x, p, ay, az, ey, ez = _inputs(500, k, bad)
    g = pic.Pic(pic.Config.from_workload(w, precision=precision), x, p, ay, az, ey, ez)
    out = torch.zeros(w.nx, dtype=torch.float64, device="cuda")
    g.deposit(pic.PIC_DEP_CHARGE, None, out)
    assert np.count_nonzero(np.isnan(out.cpu().numpy())) == k + 1
    assert not np.any(np.isfinite(g.state_numpy()["ex"]))
    assert np.isnan(g.energy()["ex"])
    g.close()


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("warm", [0, 1])
def test_2d_substep_reports_positions_that_are_not_finite(bad, warm):
    """Device arrays, which pic2d_init takes without a look at them."""
    from paper_2203_06513_gb300 import pic2d as P2
    n, M1, M2, L1, L2 = 300, 6, 5, 4.0, 3.0
    rng = np.random.default_rng(3)
    x = np.column_stack([rng.uniform(0, L1, n), rng.uniform(0, L2, n)])
    x[11, 1] = bad
    f = 0.05 * rng.normal(0, 1, (3, M1 * M2))
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, rng.normal(0, 0.2, (n, 2)), *f)]
    lib, h, it = P2._lib(), ctypes.c_void_p(), ctypes.c_int32()
    cfg = P2.Config2D(L1, L2, M1, M2, 3, n, L1 * L2 / n, 0.1, warm=warm).c()
    dp = ctypes.POINTER(ctypes.c_double)
    assert lib.pic2d_init(ctypes.byref(cfg), *(ctypes.cast(ctypes.c_void_p(t.data_ptr()), dp) for t in dev),
                          pic.PIC_MEM_DEVICE, None, ctypes.byref(h)) == 0
    assert lib.pic2d_substep1(h, ctypes.byref(it)) == pic.PIC_ERR_NUMERIC
    lib.pic2d_destroy(h)


@pytest.mark.parametrize("precision", FORMS)
@pytest.mark.parametrize("no_graph", [False, True])
def test_a_marker_that_goes_bad_in_a_later_sweep(precision, no_graph, monkeypatch):
    """A potential that is NaN in a few cells: no marker starts there, and the iterate of the
    second sweep walks into them.  Every block of the one-kernel step has to stop with that
    sweep (a block that went on alone would wait at its barrier for seconds)."""
    if no_graph:
        monkeypatch.setenv("PIC_NO_GRAPH", "1")
    nx, k, n, L = 256, 3, 20003, 8.0
    dx = L / nx
    x = (np.arange(n) + 0.5) / n * 0.5 * L          # cells 0 .. 127; node 131 reaches cells 131 .. 134
    p = np.zeros(n)
    p[-64:] = 3.0                                   # to the right by 0.95 dt = 7.6 cells
    ay = np.full(nx, 0.01)
    ay[131] = np.nan
    z = np.zeros(nx)
    for _ in range(10):
        g = pic.Pic(pic.Config(L, nx, k, n, L / n, 8 * dx, precision=precision), x, p, ay, z)
        with pytest.raises(pic.PicError) as e:
            g.step(3)
        assert e.value.code == pic.PIC_ERR_NUMERIC
        g.close()
