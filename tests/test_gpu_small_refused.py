"""Small plasmas where the device does not hold the grid of their one kernel at once: the
cooperative launch is refused, here by a stand-in for that call (a preloaded library in a
process of its own), and the steps go on as host loops and graphs with the same result."""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(shutil.which("gcc") is None, reason="needs gcc")]

SHIM = r"""
int refused;
int cudaLaunchCooperativeKernel(const void *f, ...) { ++refused; return 720; }   /* cudaErrorCooperativeLaunchTooLarge */
"""

STEPS = r"""
import ctypes, os, sys
import numpy as np
from paper_2203_06513_gb300 import inputs as I, pic
shim = ctypes.CDLL(sys.argv[1])
for kw in (dict(sort_every=2), dict(precision=pic.PIC_FP32, warm_start=1, warm_field=1), dict(hbar=0.1)):
    w = I.Workload("r", nx=48, degree=3, np=2003, vth=0.2, pump=0.2, seed=5)
    x, p = I.particles(w)
    spin = None
    if "hbar" in kw:
        s = np.random.default_rng(1).normal(size=(3, w.np))
        spin = tuple(np.ascontiguousarray(v) for v in s / np.linalg.norm(s, axis=0))
    cfg = pic.Config.from_workload(w, **kw)
    states = []
    for no_graph in (False, True):
        os.environ.pop("PIC_NO_GRAPH", None)
        if no_graph:
            os.environ["PIC_NO_GRAPH"] = "1"
        before = ctypes.c_int.in_dll(shim, "refused").value
        g = pic.Pic(cfg, x, p, *I.fields(w), spin=spin)
        its = [g.step(1), g.step(4)]
        assert sum(a for a, _ in its) >= 5
        assert ctypes.c_int.in_dll(shim, "refused").value - before == (0 if no_graph else 1)   # asked once
        states.append(g.state_numpy())
        g.close()
    a, b = states
    tol = 1e-11 if cfg.precision == pic.PIC_FP64 else 1e-5     # rounding order of the same iteration
    d = np.mod(a["x"] - b["x"] + 0.5 * w.L, w.L) - 0.5 * w.L
    assert np.max(np.abs(d)) / w.L <= tol
    for key in b:
        if key != "x":
            assert np.max(np.abs(a[key] - b[key])) <= tol * max(np.max(np.abs(b[key])), 1e-2), key
print("steps ok")
"""


def test_a_refused_cooperative_launch_goes_on_as_graphs(tmp_path):
    src, shim = tmp_path / "shim.c", tmp_path / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(shim), str(src)], check=True)
    env = dict(os.environ, LD_PRELOAD=str(shim), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", STEPS, str(shim)], env=env, cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "steps ok" in r.stdout, r.stderr[-2000:]
