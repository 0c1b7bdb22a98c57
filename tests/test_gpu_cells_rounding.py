"""Pairs within one rounding of the radius, in the cell lists' packed test.

Each axis' square is rounded before it is added, so the squared distance of a
pair may be exactly the threshold (no edge) where a contracted multiply-add
would fall one unit below it (an edge).  The radius is chosen so that a pair of
the graph's own samples is such a pair, whichever square would be contracted,
and the rows must be those of a plain FP32 evaluation (no tolerance).
"""
import numpy as np
import pytest
import torch

from paper_1705_02403_gb300 import _native as N
from paper_1705_02403_gb300 import envgen
from paper_1705_02403_gb300.planner import BatchPlanner, Planner

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

F = np.float32


def squares(X, i, j):
    t = [x[j] - x[i] for x in X]
    return t, [v * v for v in t]


def contracted(t, q):
    """Every sum of the squares in which a square is not rounded before its addition."""
    def fma(a, c):
        return (a.astype(np.float64) * a + c).astype(F)
    first = [fma(t[0], q[1]), fma(t[1], q[0])]
    if len(t) == 2:
        return first
    return [f + q[2] for f in first] + [fma(t[2], f) for f in first + [q[0] + q[1]]]


def deciding_radii(X, count):
    """Radii r = sqrt(d2) of pairs whose d2 is the least float with that root and every contracted d2 is below it."""
    i, j = np.triu_indices(X.shape[1], 1)
    t, q = squares(X, i, j)
    d2 = sum(q[1:], q[0])
    ok = (d2 > F(0.05 ** 2)) & (d2 < F(0.1 ** 2)) & (np.sqrt(np.nextafter(d2, F(0))) < np.sqrt(d2))
    for c in contracted(t, q):
        ok &= c < d2
    at = np.nonzero(ok)[0]
    assert len(at) >= count
    return [np.sqrt(d2[k]) for k in at[:count]]


def exact_rows(X, r):
    n = X.shape[1]
    rows = []
    for a in range(0, n, 512):
        i = np.arange(a, min(n, a + 512))
        t, q = squares(X, i[:, None], np.arange(n)[None])
        near = np.sqrt(sum(q[1:], q[0])) < r
        near[np.arange(len(i)), i] = False
        rows += [np.nonzero(v)[0] for v in near]
    return rows


def check(row, col, X, r):
    want = exact_rows(X, F(r))
    assert np.array_equal(np.diff(row), [len(w) for w in want])
    assert np.array_equal(col, np.concatenate(want))


@pytest.mark.parametrize("which", range(3))
@pytest.mark.parametrize("d", [2, 3])
def test_cells_round_every_square(d, which):
    def build(r):
        pb = envgen.geometric(31, d=d, n=3000, nbox=5, r=float(r), lam=0.5)
        v = Planner(pb).build(debug_flags=N.GMT_DEBUG_PAIRS_CELLS).view()
        return v.X.cpu().numpy(), v.out_row.cpu().numpy(), v.out_col[:v.E].cpu().numpy()
    r = deciding_radii(build(0.08)[0], 3)[which]
    X, row, col = build(r)
    check(row, col, X, r)


def test_batched_cells_round_every_square():
    # nodes 2939 and 11376 of this query are such a pair at its own radius
    pb = envgen.geometric(74179, d=2, n=11591, nbox=13, r=0.0, lam=0.5)
    bp = BatchPlanner([pb])
    bp.plan()
    v = bp.view(0)
    check(v["out_row"].cpu().numpy(), v["out_col"].cpu().numpy(), v["X"].cpu().numpy(), v["r"])
