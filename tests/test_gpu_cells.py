"""The sweeps' per-cell polynomials and moment windows against the FP64 oracle at the
sizes where they can go wrong: odd and tiny grids, fewer markers than a warp or than
cells, markers never sorted again, paths over many cells and around the box, markers
piled into one cell, with and without the z component.

Tolerances: those of the parity tests for a few steps (both sides solve the same fixed
point to 1e-13 and differ in rounding order; the FP32 form carries about 2^-24 per
marker and step)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2203_06513_gb300 import inputs as I
from paper_2203_06513_gb300 import pic

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")

#       nx   k  markers   dt  vth  sort  z
SHAPES = [(33, 3, 2001, 0.05, 0.1, 0, True),
          (17, 2, 515, 0.05, 0.3, 2, False),
          (255, 5, 4099, 0.05, 0.15, 1, True),
          (8, 3, 33, 0.3, 0.5, 0, True),
          (9, 4, 1000, 0.5, 0.5, 1, False),
          (250, 3, 3000, 0.3, 0.8, 0, True),     # paths over several cells, unsorted
          (127, 5, 31, 0.1, 0.2, 0, False),
          (64, 4, 20011, 0.05, 0.1, 2, True),
          (128, 3, 3002, 0.05, 0.1, 1, False),   # one tile of sort keys, then one and a few
          (129, 2, 3003, 0.05, 0.1, 1, True)]


def _check(st, s, L, tol_x, tol):
    d = np.mod(st["x"] - s.x + 0.5 * L, L) - 0.5 * L
    assert np.max(np.abs(d)) / L <= tol_x
    for key in ("p", "ex", "ey", "ez", "ay", "az"):
        ref = getattr(s, key)
        assert np.max(np.abs(st[key] - ref)) <= tol * max(np.max(np.abs(ref)), 1e-3), key


# the float form's iterates stall above the stopping rule on a handful of markers or
# large steps, so it is checked on the denser shapes
@pytest.mark.parametrize("shape,precision", [(s, pic.PIC_FP64) for s in SHAPES] +
                         [(s, pic.PIC_FP32) for s in SHAPES if s[2] >= 2000 and s[3] <= 0.05])
def test_steps_at_awkward_shapes(shape, precision):
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
    cfg = pic.Config.from_workload(w, precision=precision, sort_every=sort, max_iter=200,
                                   warm_start=pic.PIC_WARM_EXPLICIT, warm_field=1)
    g = pic.Pic(cfg, x, p, ay, az, ey, ez)
    steps = 3
    for _ in range(steps):
        s = orc.step(s)
    g.step(steps)
    _check(g.state_numpy(), s, w.L, *((1e-11, 1e-10) if precision == pic.PIC_FP64 else (1e-5, 1e-4)))
    if precision == pic.PIC_FP64:
        assert g.energy()["gauss"] < 1e-12
    g.close()


@pytest.mark.parametrize("precision", [pic.PIC_FP64, pic.PIC_FP32])
@pytest.mark.parametrize("n", [1, 4099, (1 << 22) + 1, 5 * (1 << 20) + 77])
def test_device_state_equals_host_state(n, precision):
    """pic_get_state into device arrays (one launch, or dealt into buckets for many
    markers) gives the bits of the host copy, for all members and for p alone."""
    import torch
    nx, k = 64, 3
    g = torch.Generator(device="cuda").manual_seed(n)
    L = 4 * np.pi
    x = torch.rand(n, dtype=torch.float64, device="cuda", generator=g) * L
    p = 0.1 * torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    ay = 0.1 * torch.ones(nx, dtype=torch.float64, device="cuda")
    sim = pic.Pic(pic.Config(L, nx, k, n, L / n, 0.05, precision=precision, sort_every=1), x, p, ay, 0.5 * ay)
    ref = sim.state_numpy()
    dev = {q: torch.full((v.size,), float("nan"), dtype=torch.float64, device="cuda") for q, v in ref.items()}
    sim.get_state(**dev)
    for q, v in ref.items():
        np.testing.assert_array_equal(dev[q].cpu().numpy(), v, err_msg=q)
    only = torch.empty(n, dtype=torch.float64, device="cuda")
    sim.get_state(p=only)
    np.testing.assert_array_equal(only.cpu().numpy(), ref["p"])
    sim.close()


@pytest.mark.parametrize("n,k,kw", [
    (1, 3, {}), (31, 2, dict(warm_start=1, warm_field=1)), (33, 5, dict(splitting=1)),
    (5003, 4, dict(sort_every=2, warm_start=1)), (38912, 3, dict(warm_start=1, warm_field=1, sort_every=3)),
    (38913, 3, dict(warm_start=1, warm_field=1)), (4001, 3, dict(splitting=1, warm_start=1, warm_field=1)),
    (2003, 3, dict(hbar=0.1)), (2003, 2, dict(hbar=0.1, sort_every=1)),
    (40001, 3, dict(hbar=0.1)), (65537, 5, dict(hbar=0.1, sort_every=2))])
def test_one_kernel_steps_equal_host_loops(n, k, kw, monkeypatch):
    """Steps of a small plasma (one cooperative kernel, or just above its limit the graph)
    against the same steps driven from the host: the same iteration, so rounding order
    apart the same state and sweep counts."""
    w = I.Workload("s", nx=50, degree=k, np=n, vth=0.2, pump=0.2, seed=n)
    x, p = I.particles(w)
    ay, az, ey, ez = I.fields(w)
    az = 0.05 * np.random.default_rng(k).normal(size=w.nx)
    spin = None
    if "hbar" in kw:
        s = np.random.default_rng(n).normal(size=(3, n))
        spin = tuple(np.ascontiguousarray(v) for v in s / np.linalg.norm(s, axis=0))
    cfg = pic.Config.from_workload(w, **kw)
    a = pic.Pic(cfg, x, p, ay, az, ey, ez, spin=spin)
    got_it = a.step(5)
    got = a.state_numpy()
    monkeypatch.setenv("PIC_NO_GRAPH", "1")
    b = pic.Pic(cfg, x, p, ay, az, ey, ez, spin=spin)
    ref_it = b.step(5)
    ref = b.state_numpy()
    assert max(abs(got_it[0] - ref_it[0]), abs(got_it[1] - ref_it[1])) <= 1
    d = np.mod(got["x"] - ref["x"] + 0.5 * w.L, w.L) - 0.5 * w.L
    assert np.max(np.abs(d)) / w.L < 1e-12
    for key in ref:
        if key != "x":
            assert np.max(np.abs(got[key] - ref[key])) <= 1e-11 * max(np.max(np.abs(ref[key])), 1e-2), key
    a.close()
    b.close()


def test_one_kernel_steps_report_no_convergence():
    w = I.Workload("n", nx=32, degree=3, np=1000, pump=0.2)
    x, p = I.particles(w)
    g = pic.Pic(pic.Config.from_workload(w, max_iter=1, tol=1e-30), x, p, *I.fields(w))
    with pytest.raises(pic.NoConvergence):
        g.step(3)
    g.close()


# rows of the scratch: 32 replicas, fewer than 32 blocks, 2 replicas, one replica; paths of several laps
@pytest.mark.parametrize("nx,k,n,reach", [(8, 3, 900, 64.0), (33, 5, 1, 0.3), (100, 2, 700, 0.5), (1000, 4, 12000, 2.5),
                                          (4099, 5, 900, 1.0), (8192, 4, 700, 20.0)])
def test_noalloc_replicas_vs_oracle(nx, k, n, reach):
    """The handle-free deposit at its replica counts; half of the markers in one cell.
    Double sums on both sides: 1e-13 of w sum |disp|, as for the handle's deposit."""
    import ctypes
    import torch
    L = 4 * np.pi
    dx, w = L / nx, L / n
    rng = np.random.default_rng(nx + k)
    x = rng.uniform(0, L, n)
    x[: n // 2] = (nx // 2 + rng.random(n // 2)) * dx
    x[-1] = -3.25 * L                                              # wrapped into the box
    disp = rng.uniform(-reach, reach, n) * dx
    xd, dd = torch.from_numpy(x).cuda(), torch.from_numpy(disp).cuda()
    out = torch.full((nx,), float("nan"), dtype=torch.float64, device="cuda")
    ptr = [ctypes.c_void_p(t.data_ptr()) for t in (xd, dd, out)]
    f = pic.load().pic_deposit_current_noalloc
    f.argtypes = [ctypes.c_double, ctypes.c_int32, ctypes.c_int32, ctypes.c_int64, ctypes.c_double] + [ctypes.c_void_p] * 4
    assert f(L, nx, k, n, w, *ptr, None) == 0
    want = np.zeros(nx)
    if n <= 1000:
        for xa, da in zip(x, disp):
            want += w * O.path_integral(k, nx, dx, float(xa), float(xa + da))[1]
    else:                                                          # the handle's deposit
        ay = np.zeros(nx)
        g = pic.Pic(pic.Config(L, nx, k, n, w, 8 * dx), np.mod(x, L), np.zeros(n), ay, ay)
        ref = torch.zeros(nx, dtype=torch.float64, device="cuda")
        g.deposit(pic.PIC_DEP_CURRENT, dd, ref)
        want = ref.cpu().numpy()
        g.close()
    assert np.max(np.abs(out.cpu().numpy() - want)) < 1e-13 * w * np.sum(np.abs(disp))


#                         M1  M2  k  np   vth  dt   spin
@pytest.mark.parametrize("M1,M2,k,n,vth,dt,spin", [
    (1, 11, 3, 40, 0.2, 0.1, False), (5, 1, 2, 33, 0.2, 0.1, True), (13, 9, 5, 300, 0.2, 0.1, False),
    (40, 3, 3, 200, 1.5, 0.12, True),                              # paths over more than a cell
    (9, 10, 4, 257, 0.1, 0.02, True), (6, 7, 2, 1, 0.5, 0.05, False)])
def test_2d_awkward_shapes(M1, M2, k, n, vth, dt, spin):
    """Subsystem I in two dimensions against the oracle where blocks, cells and paths have
    edges; half of the markers in one cell, some on knots.  Both sides stop at the same
    increment: 1e-10, as in the 2D parity tests."""
    from oracle import oracle2d as O2
    from paper_2203_06513_gb300 import pic2d as P2
    rng = np.random.default_rng(100 * M1 + M2)
    L1, L2 = 4.0, 3.0
    x = np.column_stack([rng.uniform(0, L1, n), rng.uniform(0, L2, n)])
    x[: n // 2] = (np.array([M1 // 2, M2 // 2]) + rng.random((n // 2, 2))) * [L1 / M1, L2 / M2]
    x[-1] = [0.0, (M2 - 1) * L2 / M2]
    p = rng.normal(0, vth, (n, 2))
    a, ex, ey, bz = (0.05 * rng.normal(0, 1, M1 * M2) for _ in range(4))
    s = rng.normal(0, 1, (n, 3))
    s /= np.linalg.norm(s, axis=1, keepdims=True)
    cfg = P2.Config2D(L1, L2, M1, M2, k, n, L1 * L2 / n, dt)
    orc = O2.Oracle2D(L1, L2, M1, M2, k, w=L1 * L2 / n, dt=dt)
    if spin:
        cfg.hbar = orc.hbar = 0.1
    g = P2.Pic2D(cfg, x, p, ex, ey, a)
    if spin:
        g.set_spin(s, bz)
    sx, sp, sex, sey = x, p, ex, ey
    for _ in range(2):
        sx, sp, sex, sey, it = orc.substep1(sx, sp, sex, sey, a, s=s if spin else None, bz=bz if spin else None)
        assert abs(g.substep1() - it) <= 1
    st = g.state()
    d = np.abs(np.mod(st["x"] - sx + 0.5 * np.array([L1, L2]), [L1, L2]) - 0.5 * np.array([L1, L2]))
    assert np.max(d / [L1, L2]) < 1e-10
    for got, ref in ((st["p"], sp), (st["ex"], sex), (st["ey"], sey)):
        assert np.max(np.abs(got - ref)) <= 1e-10 * max(np.max(np.abs(ref)), 1e-3)
    g.close()


def test_2d_large_state_copy():
    """A state larger than one copy piece comes back to pageable memory whole."""
    from paper_2203_06513_gb300 import pic2d as P2
    n, L1, L2 = 700001, 4.0, 3.0
    rng = np.random.default_rng(7)
    x = np.column_stack([rng.uniform(0, L1, n), rng.uniform(0, L2, n)])
    p = rng.normal(0, 0.1, (n, 2))
    f = np.zeros(30)
    g = P2.Pic2D(P2.Config2D(L1, L2, 6, 5, 3, n, L1 * L2 / n, 0.1), x, p, f, f, f)
    st = g.state()
    np.testing.assert_array_equal(st["p"], p)
    assert np.max(np.abs(st["x"] - x)) < 4e-15                      # cell + offset, a few roundings of L
    g.close()


@pytest.mark.parametrize("nx,k,n", [(65, 2, 1), (65, 3, 3001), (40, 5, 2050)])
def test_scaled_moments_of_uneven_fields(nx, k, n, monkeypatch):
    """The double form's sweeps (driven from the host) on potentials that differ by ten
    orders of magnitude between neighbouring nodes, markers in no order: a warp raises its
    scale many times.  Against the oracle to the parity tests' tolerances."""
    monkeypatch.setenv("PIC_NO_GRAPH", "1")
    w = I.Workload("u", nx=nx, degree=k, np=n, dt=0.02, vth=0.1, pump=0.1, seed=nx + k)
    x, p = I.particles(w)
    _, _, ey, ez = I.fields(w)
    rng = np.random.default_rng(n)
    ay, az = (0.1 * rng.choice([-1, 1], nx) * 10.0 ** rng.uniform(-10, 0, nx) for _ in range(2))
    orc = O.Oracle(w.L, nx, k, w.weight, w.dt, w.tol, 200)
    s = O.initial_state(orc, x, p, ay, az, ey, ez)
    g = pic.Pic(pic.Config.from_workload(w, sort_every=0, max_iter=200), x, p, ay, az, ey, ez)
    for _ in range(2):
        s = orc.step(s)
    g.step(2)
    _check(g.state_numpy(), s, w.L, 1e-11, 1e-10)
    g.close()
