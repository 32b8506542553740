"""Moments of the double form summed as scaled integers: a weak field beside a strong one
keeps its relative accuracy."""
import numpy as np
import pytest

from paper_2203_06513_gb300 import pic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _values(k, t):
    """N^k(r + t), r = 0 .. k, by the recursion over the degree."""
    v = [np.ones_like(t)]
    for n in range(1, k + 1):
        low, v = v, []
        for r in range(n + 1):
            a = (t + r) * low[r] if r < n else 0.0
            b = (n + 1 - r - t) * low[r - 1] if r > 0 else 0.0
            v.append((a + b) / n)
    return v


@pytest.mark.parametrize("z", [False, True])
@pytest.mark.parametrize("k", [2, 3, 4, 5])
def test_weak_fields_keep_their_digits(k, z):
    """The susceptibility deposit on a potential that is 1e10 times smaller in every other
    16 cells; a warp's markers (some 200, 100 a cell) cross from one to the other.  Nodes
    that see weak cells alone are sums of some 400 positive terms: a few roundings of 2^-53
    each, 1e-13 relative.  Positions are exact multiples of the cell width 2^-8."""
    nx, n, dx = 4096, 400_000, 2.0 ** -8
    rng = np.random.default_rng(k)
    cell = rng.integers(0, nx, n)
    t = rng.integers(1, 2 ** 30, n) * 2.0 ** -30
    p = rng.normal(0, 0.5, n)
    weak = (np.arange(nx) // 16) % 2 == 1
    a = [np.where(weak, 1e-10, 1.0) * rng.uniform(0.5, 1.0, nx) for _ in range(4)]
    if not z:
        a[1], a[3] = np.zeros(nx), np.zeros(nx)
    g = pic.Pic(pic.Config(nx * dx, nx, k, n, 1.0, 0.5 * dx), (cell + t) * dx, p, a[0], a[1])
    out = torch.zeros(2 * nx, dtype=torch.float64, device="cuda")
    g.deposit(pic.PIC_DEP_SUSCEPT, torch.from_numpy(np.concatenate(a[2:])).cuda(), out)
    got = out.cpu().numpy().reshape(2, nx)
    g.close()
    v = _values(k, t)
    node = [(cell - r) % nx for r in range(k + 1)]
    A = [sum(c[j] * w for j, w in zip(node, v)) for c in a]
    G = np.sqrt(1 + p * p + A[0] ** 2 + A[1] ** 2) + np.sqrt(1 + p * p + A[2] ** 2 + A[3] ** 2)
    # node j sees the cells j .. j + k, a cell the nodes c - k .. c
    alone = np.all([np.roll(weak, s) for s in range(-k, k + 1)], axis=0)
    assert np.count_nonzero(alone) >= nx // 8
    for c in range(2 if z else 1):
        ref = sum(np.bincount(j, (A[c] + A[2 + c]) * w / G, nx) for j, w in zip(node, v))
        assert np.max(np.abs(got[c] - ref)[alone] / ref[alone]) < 1e-13
        assert np.max(np.abs(got[c] - ref)) < 1e-13 * np.max(ref)
