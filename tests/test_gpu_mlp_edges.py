"""The training kernel of the warm-start network at batches where its tiles have edges:
one sample, a ragged tile, more tiles than resident blocks, against the float64
reference.  Tolerances: those of the training gradient's parity test (fp32 sums)."""
import numpy as np
import pytest

from oracle import mlp as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 31, 33, 4096, 30001])
def test_training_gradient_at_ragged_batches(B):
    torch = pytest.importorskip("torch")
    from paper_2203_06513_gb300 import pic
    rng = np.random.default_rng(B)
    theta = (R.init(2) + 0.05 * rng.normal(size=R.N_PARAMS)).astype(np.float32)
    norm = np.array([0.5, 0, 0, 0, 0, 0, 2, 5, 20, 5, 5, 10, 0.7, 1.3], np.float32)
    X = np.column_stack([rng.random(B), rng.normal(0, 0.2, B), rng.normal(0, 0.05, B),
                         rng.normal(0, 0.2, B), rng.normal(0, 0.2, B), np.full(B, 0.05)]).astype(np.float32)
    T = rng.normal(size=(B, 2)).astype(np.float32)
    m = pic.Mlp(norm, theta)
    g = torch.full((R.N_PARAMS,), float("nan"), dtype=torch.float32, device="cuda")
    loss = m.grad(torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda(), g)
    Xn = (X.astype(np.float64) - norm[:6]) * norm[6:12].astype(np.float64)
    Tn = T.astype(np.float64) / norm[12:14].astype(np.float64)
    ref_loss, ref = R.loss(theta.astype(np.float64), Xn, Tn), R.grad(theta.astype(np.float64), Xn, Tn)
    err = np.max(np.abs(g.cpu().numpy() - ref)) / np.max(np.abs(ref))
    print(f"\nB {B}: gradient off by {err:.2e}, loss by {abs(loss / ref_loss - 1):.2e}")
    assert abs(loss - ref_loss) <= 1e-5 * ref_loss
    assert err <= 1e-4


@pytest.mark.parametrize("n,k,fp32", [(1, 3, False), (127, 2, False), (641, 4, False), (5001, 5, True),
                                      (100003, 3, True), (100003, 3, False)])
def test_network_start_reaches_the_fixed_point(n, k, fp32):
    """Steps from the network's proposal at partial tiles, several tiles a chain and every
    degree against steps from x^n: the same fixed point, to the tolerances of the parity
    tests."""
    pytest.importorskip("torch")
    from paper_2203_06513_gb300 import inputs as I
    from paper_2203_06513_gb300 import pic
    w = I.Workload("n", nx=51, degree=k, np=n, vth=0.1, pump=0.1, seed=n)
    x, p = I.particles(w)
    ay, az, ey, ez = I.fields(w)
    az = 0.05 * np.random.default_rng(k).normal(size=w.nx)
    norm = np.array([0.5, 0, 0, 0, 0, 0.05, 4.0, 5.0, 10.0, 3.0, 3.0, 10.0, 1.0, 1.0], np.float32)
    net = pic.Mlp(norm, (0.3 * R.init(11)).astype(np.float32))
    prec = pic.PIC_FP32 if fp32 else pic.PIC_FP64
    a = pic.Pic(pic.Config.from_workload(w, precision=prec, warm_start=pic.PIC_WARM_MLP), x, p, ay, az, ey, ez)
    net.attach(a)
    b = pic.Pic(pic.Config.from_workload(w, precision=prec), x, p, ay, az, ey, ez)
    a.step(2)
    b.step(2)
    got, ref = a.state_numpy(), b.state_numpy()
    d = np.mod(got["x"] - ref["x"] + 0.5 * w.L, w.L) - 0.5 * w.L
    assert np.max(np.abs(d)) / w.L <= (1e-5 if fp32 else 1e-11)
    for key in ("p", "ex", "ey", "ez", "ay", "az"):
        assert np.max(np.abs(got[key] - ref[key])) <= (1e-4 if fp32 else 1e-10) * max(np.max(np.abs(ref[key])), 1e-3), key
    a.close()
    b.close()
