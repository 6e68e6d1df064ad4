"""The perturbation sweep at the edges of its forms: rows at the limits of the register forms (128
and 256 entries), one observed state to all of them, the last matrix factored in shared memory and
the first that is not, vectors too long for shared memory, rows that clip or reach the absorption
floor, a given initial law, and both solves of an on-chip chain (correction and factorisation)."""
import numpy as np
import pytest

import oracle as O
from tests._util import close, max_rel
from tests.test_gpu_chain import Chain

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _counts(n, c, lengths, R, seed, flat):
    """Rows with exactly the given numbers of transient entries (cycled), over c columns; flat:
    nearly equal entries (nothing clips at small radii), else exponentials (many entries clip)."""
    rng = np.random.default_rng(seed)
    C = np.sort(rng.choice(n, c, replace=False))
    counts = np.zeros((n, n + 1), np.uint32)
    for i in range(n):
        k = min(c, lengths[i % len(lengths)])
        cols = C[(np.arange(k) + i * 7) % c] if k < c else C
        p = rng.uniform(0.9, 1.1, k) if flat else rng.exponential(1.0, k)
        counts[i, cols] = 1 + np.floor((0.9 * R - k) * p / p.sum()).astype(np.uint32)
        counts[i, n] = R - counts[i, :n].sum()
    return counts


@pytest.mark.parametrize("n,c,lengths,radius,r_min,flat,model,s", [
    (40, 1, [1], 0.05, 0.05, True, 0, None),
    (40, 2, [1, 2], 0.3, 0.2, False, 0, "some"),
    (60, 33, [1, 31, 32, 33], 0.05, 0.05, True, 0, None),
    (70, 70, [3, 64, 65], 0.05, 0.05, False, 0, None),
    (400, 160, [127, 128, 129, 160], 0.05, 0.05, True, 0, "some"),
    (400, 161, [126, 127, 128, 161], 0.05, 0.05, False, 0, None),
    (420, 300, [127, 128, 254, 255, 256, 300], 0.05, 0.05, True, 0, None),
    (420, 300, [127, 128, 254, 255, 256, 300], 0.05, 0.28, False, 0, "some"),
    (300, 64, [5, 40, 64], 0.9, 0.01, False, 0, None),
    (300, 64, [5, 40, 64], 0.5, 0.05, False, 1, None),
    (420, 300, [127, 255, 256, 300], 0.3, 0.05, False, 1, "some"),
    (300, 64, [5, 40, 64], 1e7, 0.05, False, 0, None),
    (460, 420, [257, 415, 416, 420], 0.05, 0.05, False, 0, None),
    (2560, 2550, [2, 30, 257], 0.05, 0.05, False, 0, None),
])
def test_sweep_forms(n, c, lengths, radius, r_min, flat, model, s):
    R = 6000
    counts = _counts(n, c, lengths, R, 7 * n + c, flat)
    sv = None
    if s:
        sv = np.random.default_rng(3).exponential(1.0, n)
        sv[::3] = 0.0
        sv /= sv.sum()
    ch = Chain(counts, R, 0.15, s=sv)
    assert ch.c == c
    P = 1 if c > 1000 else 3
    Q, r = O.assemble_q(counts, R, 0.15)
    cnt, pairs, hst, mx, bo = ch.sweep(2, P, radius, r_min, 19, model=model)
    ref = O.perturb_sweep(Q, r, sv, 2, P, radius, r_min, 19, keep=True, model=model)
    assert close(bo, ref.b)
    assert max_rel(mx, [ref.max_db, ref.max_lin_err, ref.max_rowsum_N]) < 1e-9
    assert cnt.tolist() == [ref.top1_changes, ref.topk_set_changes, ref.topk_order_changes]
    assert (pairs == ref.pair_flips).all() and (hst == ref.shift_hist).all()


@pytest.mark.parametrize("n", [1, 31, 257])
def test_rank_screen_keeps_the_band(n):
    """The FP32 screen of the ranking decides nothing inside the tie band: values equal, apart by
    less than the band, by a little more, tiny, zero, beyond FP32's range and negative."""
    afc = pytest.importorskip("paper_2605_14743_gb300")
    rng = np.random.default_rng(n)
    for top, sign in ((1.0, 1.0), (1e200, 1.0), (1.0, -1.0)):
        b = sign * rng.choice([0.25, 0.25 + 1e-10, 0.25 + 1e-6, 0.5, 1e-45, 0.0, top], n)
        if sign < 0.0:
            b -= 0.125
        tie = 1e-9
        tau = tie * max(b.max(), 0.0)   # the band's scale is at least 0
        d = b[:, None] - b[None, :]
        u = np.arange(n)
        before = (d > tau) | ((np.abs(d) <= tau) & (u[:, None] < u[None, :]))
        np.fill_diagonal(before, False)
        ref = before.sum(axis=0)
        rank = torch.empty(n, dtype=torch.int32, device="cuda")
        topk = torch.empty(1, dtype=torch.int32, device="cuda")
        afc.afc_rank_order(n, torch.from_numpy(b).cuda(), tie, 1, rank, topk,
                     torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert (rank.cpu().numpy() == ref).all()


def test_sweep_uses_the_solved_chain():
    """The sweep perturbs the chain that was solved, whatever has become of the counts since."""
    counts = _counts(60, 33, [1, 31, 32, 33], 6000, 5, False)
    ch = Chain(counts, 6000, 0.15)
    a = ch.sweep(0, 4, 0.05, 0.05, 19)
    ch.counts.zero_()
    b = ch.sweep(0, 4, 0.05, 0.05, 19)
    assert all((x == y).all() for x, y in zip(a, b))
