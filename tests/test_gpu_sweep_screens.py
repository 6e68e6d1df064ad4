"""The FP32 screens of the perturbation sweep decide nothing that FP64 decides otherwise: rows whose
absorption ends just below the floor, rows that lose nearly all of their transient mass."""
import numpy as np
import pytest

import oracle as O
from tests._util import close, max_rel
from tests.test_gpu_chain import Chain

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

R = 4_000_000_000   # counts of one part in 4e9: entries can be placed to 2.5e-10
SEED = 19


def _shifts(i, p, cols, radius):
    """The l1 model's shifts of row i on its columns (the absorbing one last)."""
    z = np.array([int(O.philox4x32([j, i, p, 1], [SEED, 0])[0]) - 2 ** 31 for j in cols], np.float64)
    d = z - z.mean()
    return d * radius / np.abs(d).sum()


def _row(n, cols, q_abs):
    """A count row: absorption q_abs, the rest spread evenly over the columns."""
    row = np.zeros(n + 1, np.uint32)
    row[cols] = int((1.0 - q_abs) * R) // len(cols)
    row[n] = R - int(row.sum(dtype=np.int64))
    return row


def _sweep(counts, p, radius, r_min):
    ch = Chain(counts, R, 0.0)
    Q, r = O.assemble_q(counts, R, 0.0)
    cnt, pairs, hst, mx, bo = ch.sweep(p, 1, radius, r_min, SEED)
    ref = O.perturb_sweep(Q, r, None, p, 1, radius, r_min, SEED, keep=True)
    return bo, mx, ref


# r_min 0.05: the floor of the workloads; below, absorptions of thousands of r_min end at the floor
@pytest.mark.parametrize("r_min,radius", [(0.05, 0.05), (1e-3, 1.5), (1e-4, 0.5), (1e-5, 0.5), (1e-6, 0.05)])
@pytest.mark.parametrize("c", [3, 200])
def test_rows_just_below_the_absorption_floor(c, r_min, radius):
    """Rows of three entries whose absorption lands 1e-9 to 1e-6 below r_min; the others absorb
    half of their mass.  The floor rescales such a row by 1 + (r_min - absorption), which shows in
    the visits and in the longest expected walk."""
    n, p = 400, 3
    rng = np.random.default_rng(c)
    counts = np.zeros((n, n + 1), np.uint32)
    below = 0
    for i in range(n):
        cols = [i % c, (i + 1) % c]
        sh = _shifts(i, p, cols + [n], radius)
        q_abs = r_min - sh[-1] - 10.0 ** rng.uniform(-9, -6) * min(1.0, radius)
        t = (1.0 - q_abs) / 2.0
        if c == 3 and i < c or sh[-1] >= 0.0 or not q_abs < 1.0 or t + min(sh[:2]) < 0.01 * t:
            q_abs = 0.5   # an ordinary row
        else:
            below += 1
        counts[i] = _row(n, cols, q_abs)
    assert below > 40
    bo, mx, ref = _sweep(counts, p, radius, r_min)
    assert close(bo, ref.b)
    assert max_rel(mx, [ref.max_db, ref.max_lin_err, ref.max_rowsum_N]) < 1e-9


def test_longest_walk_among_rows_that_cancel():
    """Every row has one transient entry that loses 0.4 of its 0.401, so the FP32 sums of the rows
    outside C are off by 1e-4 of themselves; one of them is larger by 3e-8 and holds the maximum."""
    n, radius, r_min = 7, 0.8, 0.05
    found = 0
    for p in range(4000):
        sh = [_shifts(i, p, [0, n], radius)[0] for i in range(n)]
        if max(sh) > 0.0:
            continue   # both shifts of a row are +-0.4
        for top in (1, 4):
            counts = np.zeros((n, n + 1), np.uint32)
            for i in range(n):
                counts[i] = _row(n, [0], 1.0 - (0.001 if i == 0 else 0.401 + 3e-8 * (i == top)))
            bo, mx, ref = _sweep(counts, p, radius, r_min)
            assert close(bo, ref.b)
            assert max_rel(mx, [ref.max_db, ref.max_lin_err, ref.max_rowsum_N]) < 1e-9
        found += 1
        if found == 6:
            return
    assert False, "no perturbation moves every row down"
