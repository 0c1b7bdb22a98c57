"""Asynchronous builds that take a cell list: which of them wait for the host,
and the errors they report.  A cell list that takes the place of the all-pairs
test (10500 to 12000 nodes in 2D, 14000 to 32767 in 3D) is only queued, as that
test is: a bad start is reported by the next call.  Above these sizes the build
waits, as documented, and reports it itself."""
import numpy as np
import pytest
import torch

from paper_1705_02403_gb300 import _native as N
from paper_1705_02403_gb300 import envgen
from paper_1705_02403_gb300.planner import Planner

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def planner(d, n, nbox=5):
    pl = Planner(envgen.geometric(7, d=d, n=n, nbox=nbox, r=0.0, lam=0.5)).build()
    pl.view()  # the edge arrays are there: the next builds may stay asynchronous
    return pl


def rows(pl):
    v = pl.view()
    return [t.cpu().numpy() for t in (v.out_row, v.out_col, v.out_cost)]


@pytest.mark.parametrize("d, n", [(2, 11999), (2, 20000), (3, 32767)])
def test_larger_cell_lists_report_a_bad_start_at_once(d, n):
    pl = planner(d, n)
    want = rows(pl)
    pl.pb.x_init = np.full(d, 2.0, np.float32)  # outside X
    with pytest.raises(N.GmtError, match="x_init"):
        pl.build(asynchronous=True)
    pl.pb.x_init = np.full(d, 0.05, np.float32)
    pl.build(asynchronous=True)
    assert all(np.array_equal(a, b) for a, b in zip(rows(pl), want))


@pytest.mark.parametrize("d, n", [(2, 10600), (2, 11998), (3, 14100), (3, 32766)])
def test_cell_lists_in_place_of_all_pairs_report_it_with_the_plan(d, n):
    pl = planner(d, n)
    want = rows(pl)
    pl.pb.x_init = np.full(d, 2.0, np.float32)
    pl.build(asynchronous=True)
    with pytest.raises(N.GmtError, match="x_init"):
        pl.plan()
    pl.pb.x_init = np.full(d, 0.05, np.float32)
    pl.build(asynchronous=True)
    assert all(np.array_equal(a, b) for a, b in zip(rows(pl), want))
