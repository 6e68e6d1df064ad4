"""Counts on both sides of the node limit between the global path's two kernels (settle steps up to
7,200 nodes, buckets beyond), with unit and short lengths on sparse graphs, against the oracle."""
import numpy as np
import pytest

from afc_inputs import Workload
from tests._util import oracle_counts

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
afc = pytest.importorskip("paper_2605_14743_gb300")


@pytest.mark.parametrize("n", [7200, 7201])
@pytest.mark.parametrize("w_hi,precision", [(1, "fp64"), (10, "fp32_recheck")])
def test_counts_at_the_node_limit(n, w_hi, precision):
    rng = np.random.default_rng(n + w_hi)
    ids = np.append(np.arange(0, n, 4), n - 1)   # most nodes isolated: few sources for the oracle
    i, j = rng.choice(ids, 3000), rng.choice(ids, 3000)
    keys = np.unique((np.minimum(i, j) * n + np.maximum(i, j))[i != j])
    wl = Workload("limit", n, (keys // n).astype(np.int32), (keys % n).astype(np.int32), 0.9, 1, w_hi,
                  2, precision=precision)
    q = afc.Query(wl)
    q.run_counts()
    torch.cuda.synchronize()
    ref, _ = oracle_counts(wl, 0, wl.realizations, threads=8)
    assert (q.counts.cpu().numpy().view(np.uint32) == ref).all()
