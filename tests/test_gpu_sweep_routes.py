"""Which perturbations of a sweep are corrected and which are factored, with the oracle's results either
way: moves of a few percent up to half of a row's mass are corrected."""
import numpy as np
import pytest

import oracle as O
from tests._util import close, max_rel
from tests.test_gpu_chain import Chain
from tests.test_gpu_sweep_forms import _counts

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("radius", [0.05, 0.2, 0.35, 0.5])
@pytest.mark.parametrize("n,c,lengths", [(300, 200, [120]), (420, 300, [60, 120, 250])])
def test_wide_moves_are_corrected(n, c, lengths, radius):
    R, P = 10000, 6
    counts = _counts(n, c, lengths, R, n + c, False)
    ch = Chain(counts, R, 0.15)
    Q, r = O.assemble_q(counts, R, 0.15)
    stats = torch.zeros(2, dtype=torch.int64, device="cuda")
    cnt, pairs, hst, mx, bo = ch.sweep(1, P, radius, 0.05, 19, stats=stats)
    ref = O.perturb_sweep(Q, r, None, 1, P, radius, 0.05, 19, keep=True)
    assert close(bo, ref.b, rel=1e-12)
    assert max_rel(mx, [ref.max_db, ref.max_lin_err, ref.max_rowsum_N]) < 1e-9
    assert (hst == ref.shift_hist).all()
    assert stats.cpu().numpy().tolist() == [P, 0]


@pytest.mark.parametrize("c", [1, 2, 31, 32, 33, 97, 160])
def test_factored_on_chip(c):
    """The multiplicative model's perturbations are factored in shared memory: pivots at the edges of
    a warp's rows, with rows that move (few entries, little absorption)."""
    n, R, P = 170, 6000, 5
    counts = _counts(n, c, [1, 2, 3, 40], R, c, False)
    ch = Chain(counts, R, 0.0)
    Q, r = O.assemble_q(counts, R, 0.0)
    cnt, pairs, hst, mx, bo = ch.sweep(0, P, 0.9, 0.01, 7, model=1)
    ref = O.perturb_sweep(Q, r, None, 0, P, 0.9, 0.01, 7, keep=True, model=1)
    assert close(bo, ref.b)
    assert max_rel(mx, [ref.max_db, ref.max_lin_err, ref.max_rowsum_N]) < 1e-9
    assert (hst == ref.shift_hist).all()


@pytest.mark.parametrize("c", [16, 17, 24, 25, 41])
@pytest.mark.parametrize("radius", [0.05, 0.09, 0.11, 0.5, 0.8])
def test_short_chains(c, radius):
    """Around the sizes and widths up to which a chain is factored without corrections."""
    n, R, P = 90, 6000, 5
    counts = _counts(n, c, [2, 9, c], R, c, False)
    ch = Chain(counts, R, 0.15)
    Q, r = O.assemble_q(counts, R, 0.15)
    cnt, pairs, hst, mx, bo = ch.sweep(0, P, radius, 0.05, 7)
    ref = O.perturb_sweep(Q, r, None, 0, P, radius, 0.05, 7, keep=True)
    assert close(bo, ref.b, rel=1e-12)
    assert max_rel(mx, [ref.max_db, ref.max_lin_err, ref.max_rowsum_N]) < 1e-9
    assert cnt.tolist() == [ref.top1_changes, ref.topk_set_changes, ref.topk_order_changes]
    assert (pairs == ref.pair_flips).all() and (hst == ref.shift_hist).all()
