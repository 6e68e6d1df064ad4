"""Malformed graph rows in the on-chip form (graphs of up to 240 nodes): what the other forms report or
ignore, it reports or ignores too."""
import numpy as np
import pytest

from afc_inputs import Workload, er_edges

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
afc = pytest.importorskip("paper_2605_14743_gb300")

SHARED, GLOBAL = afc.AFC_PATH_SHARED, afc.AFC_PATH_GLOBAL
N = 60


def _query(path, **kw):
    eu, ev = er_edges(N, 0.1, 4)
    return afc.Query(Workload("rows", N, eu, ev, 0.9, 1, 9, 3, seed=6, k_min=2), memory_path=path, **kw)


def _run(q):
    q.run_counts(0, 3)
    torch.cuda.synchronize()
    st = dict(zip([f[0] for f in afc.McStats._fields_], q.stats.cpu().tolist()))
    return q.counts.cpu().numpy(), st["device_error"]


@pytest.mark.parametrize("path", [SHARED, GLOBAL])
@pytest.mark.parametrize("hop", [None, 0, 1, 2])
@pytest.mark.parametrize("what", ["col", "eid"])
def test_bad_arcs_are_reported(what, hop, path):
    """An edge whose two arcs name no node (or no edge): reported in every mode, also where the arcs
    lie outside the neighbourhoods that are drawn."""
    q = _query(path, **({} if hop is None else dict(per_row=True, hop_radius=hop)))
    assert _run(q)[1] == 0
    q.stats.zero_()
    k = torch.nonzero(q.graph.eid == 5).flatten()
    assert k.numel() == 2
    (q.graph.col if what == "col" else q.graph.eid)[k] = N if what == "col" else q.graph.m
    assert _run(q)[1] == 1


@pytest.mark.parametrize("path", [SHARED, GLOBAL])
@pytest.mark.parametrize("hop", [None, 1])
def test_arcs_outside_the_rows_are_not_read(hop, path):
    """Room for one more edge behind the last row, never filled."""
    kw = {} if hop is None else dict(per_row=True, hop_radius=hop)
    ref, err = _run(_query(path, **kw))
    assert err == 0
    q = _query(path, **kw)
    tail = torch.tensor([-1, 2 * N], dtype=torch.int32, device="cuda")
    col, eid = torch.cat([q.graph.col, tail]), torch.cat([q.graph.eid, tail.flip(0)])
    q.prob.col, q.prob.eid, q.prob.m = col.data_ptr(), eid.data_ptr(), q.graph.m + 1
    q.ws_counts = torch.empty(max(afc.afc_transition_counts_workspace(q.prob), 256),
                              dtype=torch.uint8, device="cuda")
    counts, err = _run(q)
    assert err == 0 and (counts == ref).all()
