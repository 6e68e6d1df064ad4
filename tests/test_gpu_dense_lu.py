"""The device-wide FP64 LU behind the absorbing-chain solve at the edges of its panels and of its
one-panel range: factors and pivots reproduce the permuted matrix, visits and E[T] match numpy's
dense solve, with and without row swaps, and a tall panel that does not fit in shared memory."""
import numpy as np
import pytest

from afc_inputs import Workload, path_edges

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
afc = pytest.importorskip("paper_2605_14743_gb300")


def _solve(n, c, swaps, seed):
    """Random counts over c observed states; with swaps most states return to themselves almost
    surely while a few large entries sit below the diagonal, so partial pivoting moves rows."""
    rng = np.random.default_rng(seed)
    R = 4096
    C = np.sort(rng.choice(n, c, replace=False))
    cnt = rng.multinomial(R - R // 8, rng.dirichlet(np.ones(c)), size=n)
    if swaps:
        for a in range(c):
            cnt[C[a]] //= 64
            cnt[C[a], a] = 0
            cnt[C[a], a] = R - R // 16 - cnt[C[a]].sum()
        for a in range(1, c, 3):   # rows whose mass goes to an earlier state
            cnt[C[a]] //= 64
            cnt[C[a], a - 1] += R - R // 8 - cnt[C[a]].sum()
    cnt[np.arange(c) % n, np.arange(c)] += (cnt.sum(0) == 0)
    counts = np.zeros((n, n + 1), np.int64)
    counts[:, C] = cnt
    counts[:, n] = R - cnt.sum(1)
    assert counts.min() >= 0
    eu, ev = path_edges(n)
    wl = Workload("lu", n, eu, ev, 1.0, 1, 1, R, alpha=0.0 if swaps else 0.15)
    q = afc.Query(wl)
    q.counts.copy_(torch.from_numpy(counts.astype(np.int32)))
    q.run_solve()
    torch.cuda.synchronize()
    assert q.c == c
    Q = (1.0 - wl.alpha) * counts[:, :n] / R
    A = np.eye(c) - Q[np.ix_(C, C)]
    lu = q.lu[:c * c].reshape(c, c).cpu().numpy()
    piv = q.piv[:c].cpu().numpy()
    PA = A.copy()
    for k in range(c):
        assert k <= piv[k] < c
        PA[[k, piv[k]]] = PA[[piv[k], k]]
    L, U = np.tril(lu, -1) + np.eye(c), np.triu(lu)
    assert np.abs(L).max() <= 1.0 + 1e-12
    # backward error of an LU with partial pivoting: a small multiple of c eps max|U|
    assert np.abs(L @ U - PA).max() <= 4 * c * 2.3e-16 * max(1.0, np.abs(U).max())
    s = np.full(n, 1.0 / n)
    mu = np.linalg.solve((np.eye(n) - Q).T, s)
    got = q.mu.cpu().numpy()
    assert np.abs(got - mu).max() <= 1e-9 * mu.max()
    sc = q.scalars.cpu().numpy()
    assert abs(sc[0] - mu.sum()) <= 1e-9 * mu.sum()
    t = np.linalg.solve(np.eye(n) - Q, np.ones(n))
    assert abs(sc[2] - t.max()) <= 1e-9 * t.max()
    return piv


@pytest.mark.parametrize("c", [1, 2, 7, 8, 9, 31, 33, 64, 111, 112, 113, 120, 129, 257])
@pytest.mark.parametrize("swaps", [False, True])
def test_lu_at_panel_edges(c, swaps):
    piv = _solve(max(2 * c, 40), c, swaps, 10 + c)
    if swaps and c > 8:
        assert (piv != np.arange(c)).any()


def test_panel_in_place():
    """3,200 states: the first panels are too tall for shared memory and are factored in place."""
    _solve(3300, 3200, False, 5)
