"""The forms of the settle-step routine (plain and LONG: doubled distance keys, level-ordered
backward pass, two lanes per node) on both counting paths against the CPU oracle: betweenness at
1e-9, next states and counts bit-exact, at the lengths where the form changes, at the largest
lengths of the LONG form, on deep graphs whose levels do not fit the distance words or the level
counters, and where a LONG realization is redone with 64-bit path counts."""
import numpy as np
import pytest

import oracle as O  # noqa: F401  (the oracle must be importable: the checks run against it)
from afc_inputs import Workload, er_edges, grid_edges, path_edges, ws_edges
from tests._util import max_rel, oracle_realization

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
afc = pytest.importorskip("paper_2605_14743_gb300")

SHARED, GLOBAL = afc.AFC_PATH_SHARED, afc.AFC_PATH_GLOBAL


def _check(wl, R, path):
    q = afc.Query(wl, memory_path=path)
    bc = torch.empty((R, wl.n), dtype=torch.float64, device="cuda")
    nx = torch.empty((R, wl.n), dtype=torch.int32, device="cuda")
    q.run_counts(0, R, dump_bc=bc, dump_next=nx)
    torch.cuda.synchronize()
    bc, nx = bc.cpu().numpy(), nx.cpu().numpy()
    counts = np.zeros((wl.n, wl.n + 1), np.uint32)
    for r in range(R):
        _, _, _, _, obc, onx = oracle_realization(wl, r, threads=4)
        assert max_rel(bc[r], obc) < 1e-9
        assert (nx[r] == onx).all()
        counts[np.arange(wl.n), onx] += 1
    assert (q.counts.cpu().numpy().view(np.uint32) == counts).all()
    st = dict(zip([f[0] for f in afc.McStats._fields_], q.stats.cpu().tolist()))
    assert st["device_error"] == 0 and st["overflow"] == 0
    return st


@pytest.mark.parametrize("path", [SHARED, GLOBAL])
@pytest.mark.parametrize("w_hi", [1, 23, 24, 63, 64, 32767])
@pytest.mark.parametrize("family,n", [("er", 61), ("ws", 190)])
def test_forms_by_length(family, n, w_hi, path):
    eu, ev = er_edges(n, 5.0 / n, 3) if family == "er" else ws_edges(n, 6, 0.1, 4)
    _check(Workload("forms", n, eu, ev, 0.9, 1, w_hi, 3, seed=9, k_min=3), 3, path)


@pytest.mark.parametrize("path", [SHARED, GLOBAL])
@pytest.mark.parametrize("n,w_lo,w_hi", [(65, 64, 64), (66, 64, 64), (300, 64, 100),
                                         (300, 30000, 32767)])
def test_deep_paths(n, w_lo, w_hi, path):
    """Paths have a level per node: 64 and 65 of them around the level counters of the arena
    slots, 300 beyond, and with lengths near 2^15 more than the distance words have room for."""
    eu, ev = path_edges(n)
    _check(Workload("deep", n, eu, ev, 0.995, w_lo, w_hi, 2, seed=5, k_min=2), 2, path)


def test_long_form_redone_with_wide_slots():
    """A 30 x 30 grid of equal lengths 24: path counts above 2^32, so the LONG form's compact
    slots are redone with wide ones."""
    eu, ev = grid_edges(30, 30)
    st = _check(Workload("grid24", 900, eu, ev, 0.98, 24, 24, 2, seed=3), 2, SHARED)
    assert st["wide_redone"] == 2


def test_stars_and_single_arcs():
    """Nodes with one arc (no second smallest length) and a hub with equal and distinct ones."""
    n = 130
    eu, ev = np.zeros(n - 1, np.int32), np.arange(1, n, dtype=np.int32)
    for w_lo in (1, 100):
        for path in (SHARED, GLOBAL):
            _check(Workload("star", n, eu, ev, 0.95, w_lo, 100, 2, seed=2, k_min=2), 2, path)


@pytest.mark.parametrize("n,R", [(1, 3), (2, 3), (33, 700), (240, 4), (241, 4)])
@pytest.mark.parametrize("w_hi", [9, 50])
def test_small_graph_form(n, R, w_hi):
    """The on-chip form's range (240 nodes), its smallest graphs, and more realizations than CTAs
    (the others are claimed); few realizations take CTAs of more warps."""
    eu, ev = ws_edges(n, 4, 0.2, 6) if n > 4 else path_edges(n)
    _check(Workload("small", n, eu, ev, 0.85, 1, w_hi, R, seed=8, k_min=2), R, SHARED)


def test_small_dense_graph_without_room_for_the_drawn_arcs():
    """A complete graph of 170 nodes: its arcs fit on chip once, not twice."""
    from afc_inputs import complete_edges
    eu, ev = complete_edges(170)
    _check(Workload("dense", 170, eu, ev, 0.5, 1, 40, 2, seed=4), 2, SHARED)


@pytest.mark.parametrize("block", [256, 512, 1024])
def test_small_graph_block_sizes(block):
    eu, ev = er_edges(60, 0.1, 3)
    wl = Workload("blocks", 60, eu, ev, 0.9, 1, 10, 40, seed=2)
    a = afc.Query(wl, block_threads=block)
    b = afc.Query(wl, memory_path=GLOBAL)
    a.run_counts()
    b.run_counts()
    torch.cuda.synchronize()
    assert (a.counts == b.counts).all() and (a.stats[:3] == b.stats[:3]).all()
