"""The work this library is used for, as cases of its public entry points.

A case is a dict of plain values.  `listed()` names the fixed ones, `draw()` gives
more of the same ranges, `prepare()` makes what a program holds before the call
(inputs from a seed, a handle), `run()` is one pass through the public binding,
`work()` the bytes and operations a pass cannot do without, and `exact()` the same
outputs in 64 bits by plain torch, without the library.

Kinds:
  run      one plasma (pic.Pic): a burst of time steps, then the state
  ensemble independent plasmas advanced together (pic.Ensemble), then their states
  twod     subsystem I of the two-dimensional scheme (pic2d.Pic2D), then the state
  grid     the deposits and gathers of a plasma's markers at given displacements
  noalloc  the handle-free current deposit
  train    an Adam step of the warm-start network, then its gradient and inference
State and deposits of the single-precision form are returned in single precision,
the precision its markers are kept in.
"""
import ctypes
import math
import os

import numpy as np
import torch

from paper_2203_06513_gb300 import pic, pic2d

TOL = 1e-13
WARM = {"none": pic.PIC_WARM_NONE, "explicit": pic.PIC_WARM_EXPLICIT, "learned": pic.PIC_WARM_MLP}
CIRCULAR_L = 2.0 * math.pi * math.sqrt(2.0)      # the paper's box, one wavelength
L4PI = 4.0 * math.pi


def _run(**kw):
    c = {"kind": "run", "form": "fp64", "np": 20000, "nx": 128, "degree": 3, "dt": 0.05, "steps": 2, "warm": "none",
         "sort_every": 2, "strang": False, "wave": "standing", "pump": 0.1, "vth": 0.1, "hbar": 0.0}
    c.update(kw)
    return c


PAPER = dict(wave="circular", pump=math.sqrt(3.0), vth=math.sqrt(3.0 / 511.0), dt=0.02)


def listed():
    return [
        # the paper's parametric-instability run: few markers, thousands of steps, so
        # what a step costs is launches and latency
        _run(name="paper_4e3", np=4000, steps=20, sort_every=0, **PAPER),
        # the paper's spin run (hbar = 0.1)
        _run(name="paper_spin_1e4", np=10000, steps=10, sort_every=0, hbar=0.1, **PAPER),
        # a production plasma in double precision on the grid of the scale workload
        _run(name="fp64_k3_1e7", np=10_000_000, nx=2048, pump=0.2, steps=2, warm="explicit"),
        # quintic splines in double, symmetric splitting, ragged sizes
        _run(name="fp64_k5_strang", np=1_000_003, nx=1022, degree=5, pump=0.3, vth=0.05, steps=2, strang=True),
        # the scale workload: single-precision markers, explicit and learned starts
        _run(name="fp32_k3_1e8", form="fp32", np=100_000_000, nx=2048, pump=0.2, steps=4, warm="explicit"),
        _run(name="fp32_learned_1e8", form="fp32", np=100_000_000, nx=2048, pump=0.2, steps=4, warm="learned"),
        # quintic splines in single precision, half that many markers on a coarser grid
        _run(name="fp32_k5_5e7", form="fp32", np=50_000_000, nx=1024, degree=5, pump=0.1, steps=4, warm="explicit"),
        # a parameter scan: 64 plasmas of mixed sizes in one ensemble
        {"name": "ensemble_64", "kind": "ensemble", "form": "fp32", "runs": 64, "np_lo": 20000, "np_hi": 800000,
         "degree": 3, "warm": "explicit", "steps": 4},
        # the two-dimensional substep at its benchmark size
        {"name": "twod_k3_2e6", "kind": "twod", "np": 2_000_000, "M1": 64, "M2": 64, "degree": 3, "hbar": 0.0,
         "warm": 0, "steps": 2, "dt": 0.05, "vth": 0.1},
        # deposits and gathers as separate calls (coupling to another solver)
        {"name": "grid_fp32_1e7", "kind": "grid", "form": "fp32", "np": 10_000_000, "nx": 2048, "degree": 3,
         "dt": 0.05},
        # the handle-free deposit of a plugin
        {"name": "noalloc_1e6", "kind": "noalloc", "np": 1_000_000, "nx": 1000, "degree": 3, "reach": 1.5},
        # training the warm-start network at its training script's batch
        {"name": "train_4096", "kind": "train", "batch": 4096},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cells(n):
    """Grids have an even number of cells."""
    return n - n % 2


def draw(rng):
    kind = rng.choice(["run64", "run64", "run32", "run32", "run32", "spin", "learned", "ensemble", "twod", "grid",
                       "noalloc", "train"])
    k = rng.choice([2, 3, 3, 3, 4, 5])
    pump, vth = round(rng.uniform(0.01, 0.3), 4), round(rng.uniform(0.04, 0.15), 4)
    if kind == "run64":
        n = _log(rng, 2000, 2.0e6)
        nx = max(16, _cells(min(_log(rng, 48, 4000), n // 20)))
        return _run(np=n, nx=nx, degree=k, pump=pump, vth=vth, steps=2 if n > 200000 else 6,
                    warm=rng.choice(["none", "explicit"]), sort_every=rng.choice([1, 2, 3]),
                    strang=rng.random() < 0.25)
    if kind in ("run32", "learned"):
        n = _log(rng, 50000, 5.0e7)
        nx = max(32, _cells(min(_log(rng, 128, 2048), n // 100)))
        return _run(form="fp32", np=n, nx=nx, degree=k, pump=round(0.7 * pump, 4), vth=vth, steps=4,
                    warm="learned" if kind == "learned" else "explicit")
    if kind == "spin":
        return _run(np=_log(rng, 1000, 5.0e5), nx=rng.randrange(64, 400, 2), degree=k, steps=4, sort_every=0, hbar=0.1,
                    **PAPER)
    if kind == "ensemble":
        lo = _log(rng, 5000, 50000)
        return {"kind": "ensemble", "form": rng.choice(["fp32", "fp32", "fp64"]), "runs": rng.randrange(5, 49),
                "np_lo": lo, "np_hi": lo * rng.randrange(2, 12), "degree": k, "warm": "explicit", "steps": 4}
    if kind == "twod":
        return {"kind": "twod", "np": _log(rng, 2000, 4.0e5), "M1": rng.randrange(12, 64), "M2": rng.randrange(12, 64),
                "degree": k, "hbar": rng.choice([0.0, 0.1]), "warm": rng.choice([0, 1]), "steps": 2, "dt": 0.05,
                "vth": vth}
    if kind == "grid":
        n = _log(rng, 20000, 1.0e7)
        return {"kind": "grid", "form": rng.choice(["fp32", "fp64"]), "np": n, "nx": max(32, _cells(min(_log(rng, 64, 4000), n // 50))),
                "degree": k, "dt": 0.05}
    if kind == "noalloc":
        return {"kind": "noalloc", "np": _log(rng, 1000, 5.0e6), "nx": _log(rng, 32, 8192), "degree": k,
                "reach": round(rng.uniform(0.1, 6.0), 3)}
    return {"kind": "train", "batch": _log(rng, 256, 65536)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed, salt=0):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed) * 1009 + salt)
    return g


def _markers(n, L, vth, seed, eps=0.01, kappa=0.5, salt=0):
    """x with density 1 + eps cos(kappa x) (inverse CDF by Newton), p ~ N(0, vth^2)."""
    g = _gen(seed, salt)
    x = torch.rand(n, dtype=torch.float64, device=_dev(), generator=g).mul_(L)
    if eps:
        u = x.clone()
        for _ in range(4):
            x -= (x + (eps / kappa) * torch.sin(kappa * x) - u) / (1.0 + eps * torch.cos(kappa * x))
        x.remainder_(L)
        x[x >= L] = 0.0
    p = torch.randn(n, dtype=torch.float64, device=_dev(), generator=g).mul_(vth)
    return x, p


def _waves(case, nx, L, k, seed):
    """(ay, az, ey, ez): values of the wave at the Greville abscissae; the phase is the seed's."""
    ph = 0.1 * (int(seed) % 63)
    gx = (torch.arange(nx, dtype=torch.float64, device=_dev()) + 0.5 * (k + 1)) * (L / nx)
    a = case["pump"]
    if case["wave"] == "circular":
        th = 2.0 * math.pi / L * gx + ph
        return -a * torch.sin(th), a * torch.cos(th), a * torch.cos(th), a * torch.sin(th)
    z = torch.zeros_like(gx)
    return a * torch.cos(2.0 * math.pi * 4 / L * gx + ph), z, z.clone(), z.clone()


def _box(case):
    return CIRCULAR_L if case["wave"] == "circular" else L4PI


def _run_inputs(case, seed):
    L, n, nx, k = _box(case), case["np"], case["nx"], case["degree"]
    homogeneous = case["wave"] == "circular"
    x, p = _markers(n, L, case["vth"], seed, eps=0.0 if homogeneous else 0.01)
    spin = None
    if case["hbar"]:
        s = torch.randn(3, n, dtype=torch.float64, device=_dev(), generator=_gen(seed, 3))
        s /= s.norm(dim=0)
        spin = (s[0].contiguous(), s[1].contiguous(), s[2].contiguous())
    return L, x, p, _waves(case, nx, L, k, seed), spin


def _weights():
    f = np.load(os.path.join(os.path.dirname(os.path.abspath(pic.__file__)), "data", "warm_mlp.npz"))
    return f["params"], f["norm"]


def _f64(*shape):
    return torch.empty(*shape, dtype=torch.float64, device="cuda")


def _state_buffers(n, nx, spin):
    b = {"x": _f64(n), "p": _f64(n)}
    b.update({q: _f64(nx) for q in ("ex", "ey", "ez", "ay", "az")})
    if spin:
        b.update({q: _f64(n) for q in ("sx", "sy", "sz")})
    return b


def _members(case, seed):
    """Sizes of an ensemble's runs: a property of the case, not of the seed."""
    r = np.random.default_rng([case["runs"], case["np_lo"], case["np_hi"]])
    out = []
    for _ in range(case["runs"]):
        nx = int(r.choice([256, 512, 1024, 2048]))
        n = int(math.exp(r.uniform(math.log(case["np_lo"]), math.log(case["np_hi"]))))
        out.append(_run(form=case["form"], np=n, nx=max(32, _cells(min(nx, n // 50))), degree=case["degree"], warm=case["warm"],
                        steps=case["steps"], pump=float(r.uniform(0.01, 0.3)), vth=float(r.uniform(0.04, 0.15))))
    return out


def _config(c):
    L = _box(c)
    return pic.Config(L, c["nx"], c["degree"], c["np"], L / c["np"], c["dt"], tol=TOL,
                      precision=pic.PIC_FP32 if c["form"] == "fp32" else pic.PIC_FP64, warm_start=WARM[c["warm"]],
                      sort_every=c["sort_every"], splitting=pic.PIC_SPLIT_STRANG if c["strang"] else pic.PIC_SPLIT_LIE,
                      hbar=c["hbar"], warm_field=1 if c["warm"] != "none" else 0)


def _twod_inputs(case, seed):
    g = _gen(seed, 7)
    n, M1, M2, k = case["np"], case["M1"], case["M2"], case["degree"]
    x = torch.rand(n, 2, dtype=torch.float64, device=_dev(), generator=g) * L4PI
    p = torch.randn(n, 2, dtype=torch.float64, device=_dev(), generator=g) * case["vth"]
    g1 = (torch.arange(M1, dtype=torch.float64, device=_dev()) + 0.5 * (k + 1)) * (L4PI / M1)
    g2 = (torch.arange(M2, dtype=torch.float64, device=_dev()) + 0.5 * (k + 1)) * (L4PI / M2)
    ph = 0.1 * (int(seed) % 63)
    az = (0.2 * torch.outer(torch.cos(2.0 * g1 + ph), torch.cos(0.5 * g2))).reshape(-1)
    ex = (0.02 * torch.outer(torch.sin(0.5 * g1), torch.ones_like(g2))).reshape(-1)
    ey = (0.01 * torch.outer(torch.cos(0.5 * g1), torch.sin(g2))).reshape(-1)
    s = torch.randn(n, 3, dtype=torch.float64, device=_dev(), generator=g)
    s /= s.norm(dim=1, keepdim=True)
    bz = (0.1 * torch.outer(torch.cos(0.5 * g1 + ph), torch.cos(g2))).reshape(-1)
    return x, p, ex, ey, az, s, bz


def _grid_inputs(case, seed):
    c = _run(form=case["form"], np=case["np"], nx=case["nx"], degree=case["degree"], dt=case["dt"], pump=0.2)
    L, x, p, wv, _ = _run_inputs(c, seed)
    disp = (case["dt"] * p).contiguous()
    astar = (torch.cat([wv[0], wv[0]]) * 0.97).contiguous()
    return c, L, x, p, wv, disp, astar


def _train_inputs(case, seed):
    g = _gen(seed, 11)
    _, norm = _weights()
    nt = torch.from_numpy(norm).to(_dev())
    B = case["batch"]
    X = nt[:6] + torch.randn(B, 6, device=_dev(), generator=g) / nt[6:12]
    X[:, 0] = torch.rand(B, device=_dev(), generator=g)
    T = torch.randn(B, 2, device=_dev(), generator=g) * nt[12:]
    return X.contiguous(), T.contiguous(), norm


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "run":
        L, x, p, (ay, az, ey, ez), spin = _run_inputs(case, seed)
        sim = pic.Pic(_config(case), x, p, ay, az, ey, ez, spin=spin)
        st = {"kind": kind, "case": case, "sim": sim, "out": _state_buffers(case["np"], case["nx"], spin is not None)}
        if case["warm"] == "learned":
            params, norm = _weights()
            st["net"] = pic.Mlp(norm, params)
            st["net"].attach(sim)
        return st
    if kind == "ensemble":
        mem = _members(case, seed)
        ins = []
        for r, c in enumerate(mem):
            _, x, p, wv, _ = _run_inputs(c, seed * 131 + r)
            ins.append((x.cpu().numpy(), p.cpu().numpy()) + tuple(w.cpu().numpy() for w in wv))
        ens = pic.Ensemble([_config(c) for c in mem], ins)
        n, nx = sum(c["np"] for c in mem), sum(c["nx"] for c in mem)
        return {"kind": kind, "case": case, "sim": ens, "members": mem, "out": _state_buffers(n, nx, False)}
    if kind == "twod":
        x, p, ex, ey, az, s, bz = (v.cpu().numpy() for v in _twod_inputs(case, seed))
        cfg = pic2d.Config2D(L4PI, L4PI, case["M1"], case["M2"], case["degree"], case["np"], L4PI * L4PI / case["np"],
                             case["dt"], tol=TOL, hbar=case["hbar"], warm=case["warm"])
        sim = pic2d.Pic2D(cfg, x, p, ex, ey, az)
        if case["hbar"]:
            sim.set_spin(s, bz)
        return {"kind": kind, "case": case, "sim": sim}
    if kind == "grid":
        c, L, x, p, wv, disp, astar = _grid_inputs(case, seed)
        sim = pic.Pic(_config(c), x, p, *wv)
        n, nx = case["np"], case["nx"]
        out = {"rho": _f64(nx), "j": _f64(nx), "chi": _f64(2 * nx), "ex": _f64(n), "ay": _f64(n), "mean": _f64(n)}
        return {"kind": kind, "case": case, "sim": sim, "disp": disp, "astar": astar, "out": out}
    if kind == "noalloc":
        x, p = _markers(case["np"], L4PI, 1.0, seed)
        disp = (p * (case["reach"] * L4PI / case["nx"] / 6.0)).contiguous()
        lib = pic.load()
        f = lib.pic_deposit_current_noalloc
        f.argtypes = [ctypes.c_double, ctypes.c_int32, ctypes.c_int32, ctypes.c_int64, ctypes.c_double,
                      ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
        return {"kind": kind, "case": case, "f": f, "x": x, "disp": disp, "out": _f64(case["nx"])}
    X, T, norm = _train_inputs(case, seed)
    params, _ = _weights()
    return {"kind": kind, "case": case, "net": pic.Mlp(norm, params), "X": X, "T": T,
            "grad": torch.empty(pic.N_MLP_PARAMS, device="cuda"), "Y": torch.empty(X.shape[0], 2, device="cuda")}


def _in_form(case, out):
    return {k: v.float() for k, v in out.items()} if case["form"] == "fp32" else dict(out)


def run(state):
    kind, case = state["kind"], state["case"]
    if kind == "run":
        state["sim"].step(case["steps"])
        state["sim"].get_state(**state["out"])
        return _in_form(case, state["out"])
    if kind == "ensemble":
        ens, out = state["sim"], state["out"]
        ens.step(case["steps"])
        a = b = 0
        for r, c in enumerate(state["members"]):
            n, m = c["np"], c["nx"]
            ens.run(r).get_state(**{q: (out[q][a:a + n] if q in ("x", "p") else out[q][b:b + m]) for q in out})
            a, b = a + n, b + m
        return _in_form(case, out)
    if kind == "twod":
        for _ in range(case["steps"]):
            state["sim"].substep1()
        return state["sim"].state()
    if kind == "grid":
        sim, out = state["sim"], state["out"]
        sim.deposit(pic.PIC_DEP_CHARGE, None, out["rho"])
        sim.deposit(pic.PIC_DEP_CURRENT, state["disp"], out["j"])
        sim.deposit(pic.PIC_DEP_SUSCEPT, state["astar"], out["chi"])
        sim.gather(pic.PIC_FIELD_EX, out["ex"])
        sim.gather(pic.PIC_FIELD_AY, out["ay"])
        out["mean"].copy_(state["disp"])
        sim.gather(pic.PIC_FIELD_EX_PATHAVG, out["mean"])
        return _in_form(case, out)
    if kind == "noalloc":
        x, d, out = state["x"], state["disp"], state["out"]
        rc = state["f"](L4PI, case["nx"], case["degree"], case["np"], L4PI / case["np"], x.data_ptr(), d.data_ptr(),
                        out.data_ptr(), None)
        if rc:
            raise pic.PicError(rc, pic.load().pic_last_error(None).decode())
        return out
    net = state["net"]
    loss = net.train_step(state["X"], state["T"], 2e-3)
    net.grad(state["X"], state["T"], state["grad"])
    net.infer(state["X"], state["Y"])
    return {"loss": loss, "params": net.params(), "grad": state["grad"], "Y": state["Y"]}


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _step_work(c):
    """Of one pass of a run: each step reads and writes the stored markers once and
    makes at least one evaluation of each subsystem; then the state goes out."""
    n, k, fp32 = c["np"], c["degree"], c["form"] == "fp32"
    stored = 12 if fp32 else 20
    basis = 2 * k * k
    ev = 3 * basis + 14 * (k + 1) + 60
    spin = (40 + 6 * k) if c["hbar"] else 0
    out = 8 if fp32 else (16 + (24 if c["hbar"] else 0))
    return {"bytes": n * (2.0 * stored * c["steps"] + out) + 40.0 * c["nx"] * (c["steps"] + 1),
            "flops": float(n) * c["steps"] * (ev + spin)}


def work(case):
    kind = case["kind"]
    if kind == "run":
        return _step_work(case)
    if kind == "ensemble":
        w = [_step_work(c) for c in _members(case, 0)]
        return {q: sum(v[q] for v in w) for q in ("bytes", "flops")}
    if kind == "twod":
        k = case["degree"]
        return {"bytes": case["np"] * (64.0 * case["steps"] + 32.0),
                "flops": float(case["np"]) * case["steps"] * (8 * k * (k + 1) + 8 * k * k + 80)}
    if kind == "grid":
        k, s = case["degree"], 12 if case["form"] == "fp32" else 20
        o = 4 if case["form"] == "fp32" else 8
        return {"bytes": case["np"] * (s + 8.0 + 3 * o) + 32.0 * case["nx"], "flops": case["np"] * (6.0 * k * k + 16 * (k + 1))}
    if kind == "noalloc":
        k = case["degree"]
        return {"bytes": 16.0 * case["np"] + 8.0 * case["nx"], "flops": case["np"] * (2.0 * k * k + 4 * k)}
    return {"bytes": case["batch"] * 40.0 + 4.0 * 8898 * 4, "flops": case["batch"] * (7 * 17408.0)}


# ---------------------------------------------------------------------------
# exact: the scheme in plain 64-bit torch
# ---------------------------------------------------------------------------
def _basis(t, d):
    """[N^d(r + t)], r = 0..d: values of the degree-d basis functions c - r in a cell."""
    v = [torch.ones_like(t)]
    for n in range(1, d + 1):
        w = []
        for r in range(n + 1):
            a = (t + r) * v[r] / n if r < n else 0.0
            b = ((n + 1 - r) - t) * v[r - 1] / n if r > 0 else 0.0
            w.append(a + b)
        v = w
    return v


def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return [float(v) for v in x], [float(v) for v in w]


def _mass_eig(d, M, dx):
    """Eigenvalues of the periodic degree-d mass matrix."""
    xq, wq = _gauss(d + 1)
    t = torch.tensor([0.5 * (v + 1.0) for v in xq], dtype=torch.float64)
    w = torch.tensor([0.5 * v for v in wq], dtype=torch.float64)
    v = _basis(t, d)
    row = torch.zeros(M, dtype=torch.float64)
    for a in range(d + 1):
        for b in range(d + 1):
            row[(b - a) % M] += dx * float((w * v[a] * v[b]).sum())
    return torch.fft.fft(row).real.to(_dev())


def _circ(eig, v):
    return torch.fft.ifft(torch.fft.fft(v) * eig).real


def _point(tab, u, d):
    """sum_r tab[c - r] N^d(r + t) at cell coordinates u; tab (M, q)."""
    c = torch.floor(u)
    v = _basis(u - c, d)
    c = c.long()
    M = tab.shape[0]
    return sum(v[r][:, None] * tab[(c - r) % M] for r in range(d + 1))


def _path_mean(tab, u0, d, deg):
    """Mean of the degree-deg spline with coefficients tab (M, q) along u0 -> u0 + d."""
    xq, wq = _gauss(max(1, deg // 2 + 1))
    M = tab.shape[0]
    c0 = torch.floor(u0)
    t0 = u0 - c0                       # offsets from the start cell, so that short pieces keep their digits
    t1 = t0 + d
    right = d >= 0
    sg = torch.where(right, 1.0, -1.0).to(u0)
    crossed = torch.floor(t1).abs()
    pieces = int(crossed.max()) + 1
    still = d == 0
    den = torch.where(still, torch.ones_like(d), d)
    s = 0.0
    for p in range(pieces):
        o = sg * p
        a = torch.where(right, torch.maximum(t0, o), torch.minimum(t0, o + 1))
        b = torch.where(right, torch.minimum(t1, o + 1), torch.maximum(t1, o))
        h = b - a
        h = torch.where(h * sg > 0, h, torch.zeros_like(h))
        if p == 0:
            h = torch.where(crossed == 0, d, h)
        f = torch.where(still, torch.full_like(h, 1.0 if p == 0 else 0.0), h / den)
        mid = 0.5 * (a + b) - o
        c = c0 + o
        ci = c.long()
        for x, w in zip(xq, wq):
            v = _basis(mid + 0.5 * x * h, deg)
            for r in range(deg + 1):
                s = s + (0.5 * w * f * v[r])[:, None] * tab[(ci - r) % M]
    return s


def _scatter(out, u, d, val):
    c = torch.floor(u)
    v = _basis(u - c, d)
    c = c.long()
    M = out.shape[0]
    for r in range(d + 1):
        out.index_add_(0, (c - r) % M, v[r] * val)


class _Exact:
    """The 1D scheme on the whole plasma, markers taken in chunks."""

    CHUNK = 1 << 23

    def __init__(self, c, x, p, wv, spin=None):
        self.c, self.L, self.M, self.k = c, _box(c), c["nx"], c["degree"]
        self.dx = self.L / self.M
        self.w = self.L / c["np"]
        self.u, self.p = x / self.dx, p.clone()
        self.ay, self.az, self.ey, self.ez = (v.clone() for v in wv)
        self.spin = [s.clone() for s in spin] if spin else None
        M, k, dx = self.M, self.k, self.dx
        self.m0, self.m1 = _mass_eig(k, M, dx), _mass_eig(k - 1, M, dx)
        th = 2.0 * math.pi * torch.arange(M, dtype=torch.float64, device=_dev()) / M
        self.K = self.m1 * (2.0 - 2.0 * torch.cos(th)) / dx ** 2
        rho = self.charge(self.u)
        run = torch.cumsum(self.dx * (rho - dx), 0)
        dd = torch.cat([torch.zeros(1, dtype=torch.float64, device=_dev()), run[:-1]])
        self.ex = _circ(1.0 / self.m1, dd - dd.mean())

    def chunks(self):
        n = self.u.numel()
        return [slice(a, min(n, a + self.CHUNK)) for a in range(0, n, self.CHUNK)]

    def charge(self, u, val=None, deg=None):
        out = torch.zeros(self.M, dtype=torch.float64, device=_dev())
        for s in self.chunks():
            _scatter(out, u[s], self.k if deg is None else deg, self.w * (torch.ones_like(u[s]) if val is None else val[s]))
        return out

    def diff(self, a):
        return (a - torch.roll(a, 1)) / self.dx

    def sub1(self, dt):
        k, dx = self.k, self.dx
        a2 = torch.stack([self.ay, self.az], 1)
        ga = torch.stack([self.diff(self.ay), self.diff(self.az)], 1)
        gg = torch.stack([self.diff(ga[:, 0]), self.diff(ga[:, 1])], 1)
        d = torch.zeros_like(self.u)
        pk = self.p.clone()
        ek = self.ex.clone()
        rho0 = self.charge(self.u)
        hb = self.c["hbar"]
        for it in range(60):
            tab = torch.cat([(0.5 * (self.ex + ek))[:, None], ga], 1)
            inc = 0.0
            for s in self.chunks():
                u, pn, dd = self.u[s], self.p[s], d[s]
                A0, A1 = _point(a2, u, k), _point(a2, u + dd, k)
                m = _path_mean(tab, u, dd, k - 1)
                g0, g1 = torch.sqrt(1 + pn * pn + (A0 * A0).sum(1)), torch.sqrt(1 + pn * pn + (A1 * A1).sum(1))
                q = pn + dt * m[:, 0] - dt * ((A0 + A1) * m[:, 1:]).sum(1) / (g0 + g1)
                if hb:
                    D2 = _path_mean(gg, u, dd, k - 2)
                    q = q - dt * hb * (self.spin[1][s] * D2[:, 1] - self.spin[2][s] * D2[:, 0])
                g2 = torch.sqrt(1 + q * q + (A1 * A1).sum(1))
                dn = dt * (pn + q) / (g1 + g2) / dx
                inc = max(inc, float((dn - dd).abs().max()) * dx)
                d[s] = dn
                pk[s] = q
            # j_i - j_{i+1} = dx (rho1_i - rho0_i) and sum_i j_i = sum_a w d_a: the path current
            r = self.charge(self.u + d) - rho0
            run = torch.cumsum(r * dx, 0)
            j = torch.cat([torch.zeros(1, dtype=torch.float64, device=_dev()), -run[:-1]])
            j = j - j.mean() + self.w * float(d.sum()) * dx / self.M
            en = self.ex - _circ(1.0 / self.m1, j)
            einc = float((en - ek).abs().max())
            ek = en
            if it and inc < 5e-15 and einc < 5e-15:
                break
        self.u = torch.remainder(self.u + d, self.M)
        self.p, self.ex = pk, ek

    def sub2(self, dt):
        k = self.k
        P, Pm = self.m0 + dt * dt / 4 * self.K, self.m0 - dt * dt / 4 * self.K
        by = _circ(Pm, self.ey) + dt * _circ(self.K, self.ay)
        bz = _circ(Pm, self.ez) + dt * _circ(self.K, self.az)
        if self.c["hbar"]:
            dy = self.charge(self.u, self.spin[1], k - 1)
            dz = self.charge(self.u, self.spin[2], k - 1)
            gt = lambda v: (v - torch.roll(v, -1)) / self.dx  # noqa: E731
            by = by - dt * self.c["hbar"] * gt(dz)
            bz = bz + dt * self.c["hbar"] * gt(dy)
        an = torch.stack([self.ay, self.az], 1)
        ey, ez = self.ey.clone(), self.ez.clone()
        for it in range(60):
            ak = an - 0.5 * dt * torch.stack([self.ey + ey, self.ez + ez], 1)
            sy = torch.zeros(self.M, dtype=torch.float64, device=_dev())
            sz = torch.zeros_like(sy)
            for s in self.chunks():
                A0, A1 = _point(an, self.u[s], k), _point(ak, self.u[s], k)
                pp = 1 + self.p[s] ** 2
                f = self.w * (A0 + A1) / (torch.sqrt(pp + (A0 * A0).sum(1)) + torch.sqrt(pp + (A1 * A1).sum(1)))[:, None]
                _scatter(sy, self.u[s], k, f[:, 0])
                _scatter(sz, self.u[s], k, f[:, 1])
            ny, nz = _circ(1.0 / P, by + dt * sy), _circ(1.0 / P, bz + dt * sz)
            inc = max(float((ny - ey).abs().max()), float((nz - ez).abs().max()))
            ey, ez = ny, nz
            if it and inc < 5e-15:
                break
        self.ay = self.ay - 0.5 * dt * (self.ey + ey)
        self.az = self.az - 0.5 * dt * (self.ez + ez)
        self.ey, self.ez = ey, ez

    def sub3(self, dt):
        ga = torch.stack([self.diff(self.ay), self.diff(self.az)], 1)
        g = _point(ga, self.u, self.k - 1)
        r1, r2 = g[:, 1], -g[:, 0]
        s0, s1, s2 = self.spin
        nr = torch.sqrt(r1 * r1 + r2 * r2).clamp_min(1e-300)
        a, b = torch.cos(dt * nr), torch.sin(dt * nr)
        n1, n2 = r1 / nr, r2 / nr
        dot = n1 * s1 + n2 * s2
        self.spin = [s0 * a + (n1 * s2 - n2 * s1) * b,
                     s1 * a + n2 * s0 * b + n1 * dot * (1 - a),
                     s2 * a - n1 * s0 * b + n2 * dot * (1 - a)]

    def step(self):
        dt = self.c["dt"]
        if self.c["strang"]:
            self.sub1(0.5 * dt)
            self.sub2(dt)
            self.sub1(0.5 * dt)
        else:
            self.sub1(dt)
            self.sub2(dt)
            if self.spin:
                self.sub3(dt)

    def state(self):
        out = {"x": self.u * self.dx, "p": self.p, "ex": self.ex, "ey": self.ey, "ez": self.ez, "ay": self.ay, "az": self.az}
        if self.spin:
            out.update(zip(("sx", "sy", "sz"), self.spin))
        return out


def _cuts2(u0, d):
    """Parameters where the 2D paths u0 -> u0 + d cross a knot, sorted, with 0 and 1 (n, q)."""
    cols = [torch.zeros_like(d[:, 0]), torch.ones_like(d[:, 0])]
    for q in range(2):
        lo = torch.minimum(u0[:, q], u0[:, q] + d[:, q])
        hi = torch.maximum(u0[:, q], u0[:, q] + d[:, q])
        most = int((torch.ceil(hi) - 1 - torch.floor(lo)).max())
        for m in range(1, most + 1):
            kn = torch.floor(lo) + m
            s = (kn - u0[:, q]) / torch.where(d[:, q] == 0, torch.ones_like(d[:, q]), d[:, q])
            cols.append(torch.where((kn < hi) & (d[:, q] != 0), s.clamp(0.0, 1.0), torch.ones_like(s)))
    return torch.stack(cols, 1).sort(1).values


def _tensor_at(u, d1, d2, M1, M2):
    """(index, weight) pairs of the degree (d1, d2) tensor basis at the points u (n, 2)."""
    c = torch.floor(u)
    v1, v2 = _basis(u[:, 0] - c[:, 0], d1), _basis(u[:, 1] - c[:, 1], d2)
    c = c.long()
    for r1 in range(d1 + 1):
        for r2 in range(d2 + 1):
            yield ((c[:, 0] - r1) % M1) * M2 + (c[:, 1] - r2) % M2, v1[r1] * v2[r2]


def _exact_twod(case, seed):
    x, p, ex, ey, az, spin, bz = _twod_inputs(case, seed)
    n, M1, M2, k, dt = case["np"], case["M1"], case["M2"], case["degree"], case["dt"]
    dx = torch.tensor([L4PI / M1, L4PI / M2], dtype=torch.float64, device=_dev())
    w, hb = L4PI * L4PI / n, case["hbar"]
    e0 = [_mass_eig(k, M1, L4PI / M1), _mass_eig(k, M2, L4PI / M2)]
    e1 = [_mass_eig(k - 1, M1, L4PI / M1), _mass_eig(k - 1, M2, L4PI / M2)]
    eigx, eigy = torch.outer(e1[0], e0[1]), torch.outer(e0[0], e1[1])
    solve = lambda v, eig: torch.fft.ifft2(torch.fft.fft2(v.reshape(M1, M2)) / eig).real.reshape(-1)  # noqa: E731

    def grad(a, q):
        b = a.reshape(M1, M2)
        return ((b - torch.roll(b, 1, q)) / float(dx[q])).reshape(-1)

    def value(a, u, d1, d2):
        return sum(a[i] * v for i, v in _tensor_at(u, d1, d2, M1, M2))

    def quot(terms, u0, d, q, other):
        """Mean over coordinate q from u0_q by d_q of sum_t c_t * spline_t, the other fixed at `other`."""
        base = torch.stack([u0[:, 0], other] if q == 0 else [other, u0[:, 1]], 1)
        dd = torch.zeros_like(d)
        dd[:, q] = d[:, q]
        cuts = _cuts2(base, dd)
        xq, wq = _gauss(k)
        s = 0.0
        for a in range(cuts.shape[1] - 1):
            h = cuts[:, a + 1] - cuts[:, a]
            mid = 0.5 * (cuts[:, a + 1] + cuts[:, a])
            cell = torch.floor(base + mid[:, None] * dd)
            for xx, ww in zip(xq, wq):
                u = base + (mid + 0.5 * xx * h)[:, None] * dd
                u = torch.minimum(torch.maximum(u, cell), cell + (1 - 1e-15))
                for c, arr, d1, d2 in terms:
                    s = s + c * 0.5 * ww * h * value(arr, u, d1, d2)
        return s

    for _ in range(case["steps"]):
        u0 = x / dx
        d = torch.zeros_like(x)
        pk = p.clone()
        ekx, eky = ex.clone(), ey.clone()
        gx, gy = grad(az, 0), grad(az, 1)
        A0 = value(az, u0, k, k)
        pp = (p * p).sum(1)
        for it in range(60):
            ebx, eby = 0.5 * (ex + ekx), 0.5 * (ey + eky)
            du = d / dx
            xq, wq = _gauss(k)

            def walk(dv, f):
                cuts = _cuts2(u0, dv)
                for a in range(cuts.shape[1] - 1):
                    h = cuts[:, a + 1] - cuts[:, a]
                    mid = 0.5 * (cuts[:, a + 1] + cuts[:, a])
                    cell = torch.floor(u0 + mid[:, None] * dv)
                    for xx, ww in zip(xq, wq):
                        u = u0 + (mid + 0.5 * xx * h)[:, None] * dv
                        f(torch.minimum(torch.maximum(u, cell), cell + (1 - 1e-15)), 0.5 * ww * h)

            E = [torch.zeros(n, dtype=torch.float64, device=_dev()) for _ in range(2)]

            def add(u, f):
                E[0] += f * value(ebx, u, k - 1, k)
                E[1] += f * value(eby, u, k, k - 1)
            walk(du, add)
            A1 = value(az, u0 + du, k, k)
            o1, o2 = u0[:, 1] + du[:, 1], u0[:, 0]
            D1 = quot([(1.0, gx, k - 1, k)], u0, du, 0, o1)
            D2 = quot([(1.0, gy, k, k - 1)], u0, du, 1, o2)
            g0, g1 = torch.sqrt(1 + pp + A0 * A0), torch.sqrt(1 + pp + A1 * A1)
            f = dt * (A1 + A0) / (g1 + g0)
            q0, q1 = p[:, 0] + dt * E[0] - f * D1, p[:, 1] + dt * E[1] - f * D2
            if hb:
                sx, sy, sz = spin[:, 0], spin[:, 1], spin[:, 2]
                gxy = grad(gy, 0)
                q0 = q0 - dt * hb * quot([(sx, gxy, k - 1, k - 1), (-sy, grad(gx, 0), k - 2, k),
                                          (sz, grad(bz, 0), k - 2, k - 1)], u0, du, 0, o1)
                q1 = q1 - dt * hb * quot([(-sy, gxy, k - 1, k - 1), (sx, grad(gy, 1), k, k - 2),
                                          (sz, grad(bz, 1), k - 1, k - 2)], u0, du, 1, o2)
            g2 = torch.sqrt(1 + q0 * q0 + q1 * q1 + A1 * A1)
            dn = torch.stack([dt * (p[:, 0] + q0) / (g1 + g2), dt * (p[:, 1] + q1) / (g1 + g2)], 1)
            qn = torch.stack([q0, q1], 1)
            inc = max(float((dn - d).abs().max()), float((qn - pk).abs().max()))
            d, pk = dn, qn
            jx, jy = torch.zeros(M1 * M2, dtype=torch.float64, device=_dev()), torch.zeros(M1 * M2, dtype=torch.float64, device=_dev())

            def dep(u, f):
                for i, v in _tensor_at(u, k - 1, k, M1, M2):
                    jx.index_add_(0, i, w * f * d[:, 0] * v)
                for i, v in _tensor_at(u, k, k - 1, M1, M2):
                    jy.index_add_(0, i, w * f * d[:, 1] * v)
            walk(d / dx, dep)
            nx_, ny_ = ex - solve(jx, eigx), ey - solve(jy, eigy)
            inc = max(inc, float((nx_ - ekx).abs().max()), float((ny_ - eky).abs().max()))
            ekx, eky = nx_, ny_
            if it and inc < 5e-15:
                break
        x = torch.remainder(x + d, L4PI)
        p, ex, ey = pk, ekx, eky
    return {"x": x, "p": p, "ex": ex, "ey": ey}


def _net(X, P, norm):
    n = norm.double()
    h = (X.double() - n[:6]) * n[6:12]
    o = 0
    for a, b in ((64, 6), (64, 64), (64, 64), (2, 64)):
        W, c = P[o:o + a * b].reshape(a, b), P[o + a * b:o + a * b + a]
        o += a * b + a
        h = h @ W.T + c
        if a == 64:
            h = torch.relu(h)
    return h


def _exact_train(case, seed):
    X, T, norm = _train_inputs(case, seed)
    params, _ = _weights()
    nt = torch.from_numpy(norm).to(_dev())
    P = torch.from_numpy(params).to(_dev()).double().requires_grad_(True)

    def loss_grad():
        loss = ((_net(X, P, nt) - T.double() / nt[12:].double()) ** 2).sum(1).mean()
        return loss, torch.autograd.grad(loss, P)[0]
    loss, g = loss_grad()
    with torch.no_grad():          # the first Adam step: m/c1 = g, v/c2 = g^2
        P -= 2e-3 * g / (g.abs() + 1e-8)
    g1 = loss_grad()[1]
    Y = (_net(X, P, nt) * nt[12:].double()).detach()
    return {"loss": float(loss), "params": P.detach(), "grad": g1, "Y": Y}


def _exact_grid(case, seed):
    c, L, x, p, wv, disp, astar = _grid_inputs(case, seed)
    s = _Exact(c, x, p, wv)
    k, nx, dx = s.k, s.M, s.dx
    d = disp / dx
    rho = s.charge(s.u)
    run = torch.cumsum((s.charge(s.u + d) - rho) * dx, 0)
    j = torch.cat([torch.zeros(1, dtype=torch.float64, device=_dev()), -run[:-1]])
    j = j - j.mean() + s.w * float(d.sum()) * dx / nx
    an, ak = torch.stack([s.ay, s.az], 1), torch.stack([astar[:nx], astar[nx:]], 1)
    chi = torch.zeros(2, nx, dtype=torch.float64, device=_dev())
    ex, ay, mean = [], [], []
    for sl in s.chunks():
        A0, A1 = _point(an, s.u[sl], k), _point(ak, s.u[sl], k)
        pp = 1 + p[sl] ** 2
        f = s.w * (A0 + A1) / (torch.sqrt(pp + (A0 * A0).sum(1)) + torch.sqrt(pp + (A1 * A1).sum(1)))[:, None]
        _scatter(chi[0], s.u[sl], k, f[:, 0])
        _scatter(chi[1], s.u[sl], k, f[:, 1])
        ex.append(_point(s.ex[:, None], s.u[sl], k - 1)[:, 0])
        ay.append(A0[:, 0])
        mean.append(_path_mean(s.ex[:, None], s.u[sl], d[sl], k - 1)[:, 0])
    return {"rho": rho, "j": j, "chi": chi.reshape(-1), "ex": torch.cat(ex), "ay": torch.cat(ay), "mean": torch.cat(mean)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "run":
        if case["np"] * case["steps"] > 45_000_000:        # would take long
            return None
        L, x, p, wv, spin = _run_inputs(case, seed)
        s = _Exact(case, x, p, wv, spin)
        for _ in range(case["steps"]):
            s.step()
        return s.state()
    if kind == "ensemble":
        parts = []
        for r, c in enumerate(_members(case, seed)):
            _, x, p, wv, _ = _run_inputs(c, seed * 131 + r)
            s = _Exact(c, x, p, wv)
            for _ in range(c["steps"]):
                s.step()
            parts.append(s.state())
        return {q: torch.cat([v[q] for v in parts]) for q in parts[0]}
    if kind == "twod":
        return _exact_twod(case, seed)
    if kind == "grid":
        return _exact_grid(case, seed)
    if kind == "noalloc":
        x, p = _markers(case["np"], L4PI, 1.0, seed)
        M = case["nx"]
        dx = L4PI / M
        d = p * (case["reach"] * L4PI / M / 6.0) / dx
        rho = torch.zeros(M, dtype=torch.float64, device=_dev())
        one = torch.full_like(d, L4PI / case["np"])
        _scatter(rho, x / dx + d, case["degree"], one)
        _scatter(rho, x / dx, case["degree"], -one)
        run = torch.cumsum(rho * dx, 0)
        j = torch.cat([torch.zeros(1, dtype=torch.float64, device=_dev()), -run[:-1]])
        return j - j.mean() + (L4PI / case["np"]) * float(d.sum()) * dx / M
    return _exact_train(case, seed)
