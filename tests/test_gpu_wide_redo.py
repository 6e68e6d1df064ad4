"""Realizations redone with 64-bit path counts in the on-chip form, where several small CTAs share an
SM: every thread of a CTA takes the same branch after the attempt, so every realization is redone
once and the counts are the oracle's."""
import numpy as np
import pytest

from afc_inputs import Workload
from tests._util import oracle_counts

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
afc = pytest.importorskip("paper_2605_14743_gb300")


def _diamonds(k, width):
    """k diamonds in a row: hub, `width` middle nodes, hub, ..: width^k shortest paths end to end."""
    eu, ev, n = [], [], 1
    for _ in range(k):
        for a in range(width):
            eu += [n - 1, n + a]
            ev += [n + a, n + width]
        n += width + 1
    return n, np.array(eu, np.int32), np.array(ev, np.int32)


@pytest.mark.parametrize("block", [0, 256, 512, 1024])
@pytest.mark.parametrize("w,precision", [(7, "fp64"), (40, "fp64"), (40, "fp32_recheck")])
def test_small_graphs_are_redone_with_wide_slots(block, w, precision):
    """26 diamonds of 4: 4^26 = 2^52 paths of equal lengths; some middle nodes fail."""
    n, eu, ev = _diamonds(26, 4)
    assert n <= 240
    R = 1500
    wl = Workload("diamonds", n, eu, ev, 0.995, w, w, R, seed=11, k_min=3, precision=precision)
    ref, _ = oracle_counts(wl, 0, R, threads=8)
    for _ in range(3):
        q = afc.Query(wl, block_threads=block)
        q.run_counts()
        torch.cuda.synchronize()
        assert (q.counts.cpu().numpy().view(np.uint32) == ref).all()
        st = dict(zip([f[0] for f in afc.McStats._fields_], q.stats.cpu().tolist()))
        assert st["device_error"] == 0 and st["overflow"] == 0 and st["realizations"] == R
        assert st["wide_redone"] == R   # a failed edge leaves far more than 2^32 paths
