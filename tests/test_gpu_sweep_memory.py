"""The sweep's device memory: a CTA's slab of a chain whose states are all observed, and perturbations
that follow one another in a slab whose matrix was factored."""
import pytest

from tests.test_gpu_chain import Chain
from tests.test_gpu_sweep_forms import _counts

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
afc = pytest.importorskip("paper_2605_14743_gb300")


@pytest.mark.parametrize("n", [300, 1000, 1100, 2000, 9000])
def test_workspace_of_a_fully_observed_chain(n):
    """Per CTA the matrix and the C rows in FP64 and the other rows' places in FP32 (20 n^2 bytes),
    some vectors; two CTAs per SM while their slabs take at most 8 GB."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    slab = 20 * n * n + 400 * n + 16384
    ctas = sms * (2 if 2 * sms * slab <= 8 << 30 else 1)
    others = 20 * n * (n + 1) + 200 * n + 65536   # the sparse rows, the inverse, vectors
    got = afc.afc_solve_workspace(n, n)
    assert got <= ctas * slab + others


@pytest.mark.parametrize("c,radius,model", [(170, 0.9, 1), (200, 0.05, 0)])
def test_perturbations_after_one_another(c, radius, model):
    """More perturbations than CTAs: each gives what it gives alone."""
    counts = _counts(240, c, [2, 5], 6000, c, False)
    ch = Chain(counts, 6000, 0.0 if model else 0.15)
    stats = torch.zeros(2, dtype=torch.int64, device="cuda")
    P = 700
    bo = ch.sweep(0, P, radius, 0.05, 19, model=model, stats=stats)[4]
    done = stats.cpu().numpy()
    assert done.sum() == P and (done[1] > P // 2) == (model == 1)
    for p in (0, 303, 304, 305, 511, 608, P - 1):
        assert (ch.sweep(p, 1, radius, 0.05, 19, model=model)[4][0] == bo[p]).all()
