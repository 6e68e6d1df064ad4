"""The order by level of the settle-step routine at the edges of its groups of 4 x 32 nodes, where a
compact slot's counters and order entries share words: betweenness and next states of the LONG form
against the oracle, from sparse graphs (many levels, partly reached) to dense ones."""
import pytest

from afc_inputs import Workload, er_edges, ws_edges
from tests.test_gpu_step_forms import GLOBAL, SHARED, _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", [SHARED, GLOBAL])
@pytest.mark.parametrize("n", [31, 33, 97, 127, 128, 129, 160, 255, 257, 385])
def test_level_order_at_group_edges(n, path):
    for eu, ev in (ws_edges(n, 4, 0.2, n), er_edges(n, 1.5 / n, n), er_edges(n, min(0.9, 24.0 / n), n)):
        if len(eu):
            _check(Workload("levels", n, eu, ev, 0.9, 1, 200, 2, seed=n, k_min=2), 2, path)
