"""The all-pairs tiles' sum of squares, and the cell lists that replace them.

The tiles round the second axis' square and add the others to it unrounded
(first axis first).  Radii are chosen so that pairs of the graph's own samples
lie exactly on the threshold under that sum, or one rounding off it under the
sum with every square rounded; rows must be those of the tiles' sum, exactly.
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


def sums(X, i, j):
    """(the tiles' sum, every square rounded) of pairs i, j."""
    t = [x[j] - x[i] for x in X]
    q = [v * v for v in t]
    s = (t[0].astype(np.float64) * t[0] + q[1]).astype(F)
    for v in t[2:]:
        s = (v.astype(np.float64) * v + s).astype(F)
    return s, sum(q[1:], q[0])


def deciding_radii(X, near, count, rows=400):
    """Radii at which the two sums of some pair decide differently, both ways, near the given radius."""
    i, j = (v.ravel() for v in np.meshgrid(np.arange(rows), np.arange(rows, X.shape[1]), indexing="ij"))
    s, e = sums(X, i, j)
    big = np.maximum(s, e)
    ok = (s != e) & (np.abs(big - F(near) ** 2) < F(0.3) * F(near) ** 2)
    ok &= np.sqrt(np.nextafter(big, F(0))) < np.sqrt(big)
    at = [np.nonzero(ok & (s < e))[0], np.nonzero(ok & (s > e))[0]]
    assert min(len(a) for a in at) >= count
    return [np.sqrt(big[a[k]]) for k in range(count) for a in at]


def csr(v):
    return v.out_row.cpu().numpy(), v.out_col[:v.E].cpu().numpy(), v.out_cost[:v.E].cpu().numpy()


def same(a, b):
    assert all(np.array_equal(x.view(np.int32), y.view(np.int32)) for x, y in zip(a, b))


@pytest.mark.parametrize("d, n", [(d, n) for d in (2, 3, 4) for n in (1, 31, 255, 256, 512, 1300)])
def test_all_pairs_rows(d, n):
    def build(r):
        pb = envgen.geometric(31, d=d, n=n, nbox=0 if d == 4 else 5, r=float(r), lam=0.5)
        return Planner(pb).build(debug_flags=N.GMT_DEBUG_PAIRS_ALL).view()
    near = {2: 0.15, 3: 0.25, 4: 0.4}[d]
    X = build(near).X.cpu().numpy()
    for r in deciding_radii(X, near, 2) if n == 1300 else [near, 2.5]:
        v = build(r)
        X, (row, col, _) = v.X.cpu().numpy(), csr(v)
        i, j = (g.ravel() for g in np.meshgrid(np.arange(n + 1), np.arange(n + 1), indexing="ij"))
        edge = (np.sqrt(sums(X, i, j)[0]) < F(r)) & (i != j)
        assert np.array_equal(np.diff(row), np.bincount(i[edge], minlength=n + 1))
        assert np.array_equal(col, j[edge])


@pytest.mark.parametrize("d, n, batched", [(2, 10600, False), (3, 14100, False), (2, 3300, True), (3, 5100, True)])
def test_cells_that_replace_all_pairs_keep_their_rows(d, n, batched):
    def problem(r):
        return envgen.geometric(31, d=d, n=n, nbox=5, r=float(r), lam=0.5)

    def pairs(r):
        return Planner(problem(r)).build(debug_flags=N.GMT_DEBUG_PAIRS_ALL).view()
    near = 0.05 if d == 2 else 0.12
    for r in deciding_radii(pairs(near).X.cpu().numpy(), near, 2):
        if batched:
            bp = BatchPlanner([problem(r)])
            bp.plan()
            v = bp.view(0)
            got = tuple(v[k].cpu().numpy() for k in ("out_row", "out_col", "out_cost"))
        else:
            got = csr(Planner(problem(r)).build().view())
        same(got, csr(pairs(r)))


@pytest.mark.parametrize("d", [2, 3])
def test_mirrored_tiles_of_a_batch(d):
    # enough tiles for one side of the diagonal, among them ragged small queries; each alone evaluates both sides
    sizes = [1, 30, 31, 254, 255, 256, 510, 511, 512, 767, 768, 1023] + [1300] * 48
    pbs = [envgen.geometric(500 + k, d=d, n=n, nbox=5, r=0.3, lam=0.5) for k, n in enumerate(sizes)]
    bp = BatchPlanner(pbs)
    for _ in range(2):
        bp.plan()
        for k in list(range(14)) + [len(sizes) - 1]:
            v = bp.view(k)
            got = tuple(v[f].cpu().numpy() for f in ("out_row", "out_col", "out_cost"))
            same(got, csr(Planner(pbs[k]).build(debug_flags=N.GMT_DEBUG_PAIRS_ALL).view()))


@pytest.mark.parametrize("d, n", [(2, 9984), (3, 10017), (4, 10239), (4, 10240)])
def test_mirrored_tiles_of_one_graph(d, n):
    r = {2: 0.05, 3: 0.1, 4: 0.2}[d]
    pb = envgen.geometric(31, d=d, n=n, nbox=0 if d == 4 else 5, r=r, lam=0.5)
    v = Planner(pb).build(debug_flags=N.GMT_DEBUG_PAIRS_ALL).view()
    X, (row, col, _) = v.X.cpu().numpy(), csr(v)
    rows = np.r_[0:300, 5000:5200, n - 300:n + 1]
    for a in np.array_split(rows, 16):
        i, j = (g.ravel() for g in np.meshgrid(a, np.arange(n + 1), indexing="ij"))
        edge = (np.sqrt(sums(X, i, j)[0]) < F(r)) & (i != j)
        want = j[edge]
        assert np.array_equal(np.concatenate([col[row[u]:row[u + 1]] for u in a]), want)
