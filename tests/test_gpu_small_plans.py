"""The on-chip form's CTA sizes by realization count and precision: the same counts from each."""
import numpy as np
import pytest

from afc_inputs import Workload, er_edges
from tests._util import oracle_counts

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
afc = pytest.importorskip("paper_2605_14743_gb300")


@pytest.mark.parametrize("precision", ["fp64", "fp32_recheck"])
@pytest.mark.parametrize("n", [127, 128])
def test_counts_at_the_lines_of_the_cta_rule(n, precision):
    """Realizations around 16 and 8 warps' worth per SM, plain and halved (152 SMs of 32 warps)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    eu, ev = er_edges(n, 5.0 / n, n)
    for R in (2 * sms - 1, 2 * sms, 4 * sms - 1, 4 * sms, 8 * sms - 1, 8 * sms):
        wl = Workload("plans", n, eu, ev, 0.9, 1, 20, R, seed=R, precision=precision)
        q = afc.Query(wl)
        q.run_counts()
        torch.cuda.synchronize()
        ref, _ = oracle_counts(wl, 0, R, threads=16)
        assert (q.counts.cpu().numpy().view(np.uint32) == ref).all()
