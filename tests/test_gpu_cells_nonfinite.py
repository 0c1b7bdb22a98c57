"""Cell lists with a node that is not a point: a start that is not finite (a
build that does not wait reports it with the next call) and an appended sample
that has become so when a batch is replayed.  The call ends in
GMT_ERR_INVALID, the node has no edges, and the other rows are untouched.  (A
row count that takes the node itself off without its having passed its own test
is negative, and the next row then starts before the edge arrays.)"""
import numpy as np
import pytest
import torch

from paper_1705_02403_gb300 import _native as N
from paper_1705_02403_gb300 import envgen
from paper_1705_02403_gb300.planner import BatchPlanner, Planner, wrap_device

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("d, n, axis", [(2, 10600, 0), (2, 10600, 1), (3, 14100, 2)])
def test_start_that_is_no_point(d, n, axis, bad):
    pl = Planner(envgen.geometric(7, d=d, n=n, nbox=5, r=0.0)).build()
    v = pl.view()
    want = [t.cpu().numpy() for t in (v.out_row, v.out_col, v.out_cost)]
    row = wrap_device(v.raw.out_row, (v.N + 1,), "i4", pl.graph)
    good = pl.pb.x_init.copy()
    for asynchronous in (True, False):
        pl.pb.x_init = good.copy()
        pl.pb.x_init[axis] = bad
        with pytest.raises(N.GmtError, match="x_init") as e:
            pl.build(asynchronous=asynchronous)
            pl.plan()
        assert e.value.status == N.GMT_ERR_INVALID
        if asynchronous:
            torch.cuda.synchronize()
            r = row.cpu().numpy()
            assert r[0] == 0 and r[1] == 0 and (np.diff(r) >= 0).all()
            # every other row loses at most its edge to the start
            assert (np.diff(want[0])[1:] - np.diff(r)[1:] <= 1).all()
    pl.pb.x_init = good
    pl.build(asynchronous=True)
    v = pl.view()
    assert all(np.array_equal(a.cpu().numpy(), b) for a, b in zip((v.out_row, v.out_col, v.out_cost), want))


def test_appended_sample_that_is_no_point_on_replay():
    pbs = [envgen.geometric(k, d=3, n=n, nbox=5, r=0.12) for k, n in enumerate((5100, 6000))]
    extra = torch.full((2, 3, 4), 0.5, device="cuda")
    extra += 0.01 * torch.arange(4, device="cuda")
    for pb in pbs:
        pb.box_lo, pb.box_hi = pb.box_lo[:0], pb.box_hi[:0]
    bp = BatchPlanner(pbs, extra=extra, extra_count=4)
    bp.plan()
    want = [bp.view(k)["out_row"].cpu().numpy() for k in range(2)]
    extra[1, 0, 0] = float("nan")
    for _ in range(2):  # the sequence is captured, then replayed
        infos = bp.plan(allow_errors=True)
        assert infos[0]["status"] == 0 and infos[1]["status"] == N.GMT_ERR_INVALID
        assert np.array_equal(bp.view(0)["out_row"].cpu().numpy(), want[0])
        row = np.diff(bp.view(1)["out_row"].cpu().numpy())
        node = pbs[1].N  # the first appended sample
        assert row[node] == 0 and (row >= 0).all()
        assert (np.diff(want[1]) - row <= 1)[np.arange(len(row)) != node].all()
    extra[1, 0, 0] = 0.5
    bp.plan()
    assert np.array_equal(bp.view(1)["out_row"].cpu().numpy(), want[1])
