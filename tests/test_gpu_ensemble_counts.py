"""The launch count of an ensemble."""
import pytest

from paper_2203_06513_gb300 import inputs as I
from paper_2203_06513_gb300 import pic

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")


@pytest.mark.parametrize("use_graph", [True, False])
def test_a_batched_sort_counts_its_five_kernels(use_graph):
    """One run: a step is a fixed number of launches and three a sweep; a sort due after it adds
    its kernels (counts cleared, histogram, two of the scan, scatter)."""
    w = I.Workload("n", nx=64, degree=3, np=3001)
    x, p = I.particles(w)
    fixed = []
    for every in (0, 1):
        cfg = pic.Config.from_workload(w, sort_every=every)
        e = pic.Ensemble([cfg], [(x, p, *I.fields(w))], use_graph=use_graph)
        sweeps, _ = e.step(1)
        fixed.append(e.launches - 3 * int(sweeps.sum()))
        e.close()
    assert fixed[1] - fixed[0] == 5
