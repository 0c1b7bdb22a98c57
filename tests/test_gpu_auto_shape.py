"""The automatic launch shape of a handle that is built again at another size:
it is chosen for the graph the handle holds now, and the tree is the oracle's."""
import numpy as np
import pytest
import torch

from paper_1705_02403_gb300 import _native as N
from paper_1705_02403_gb300 import envgen
from paper_1705_02403_gb300.planner import Planner
from test_gpu_parity import bits, oracle_run

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("sizes", [(600, 3000), (3000, 600)])
def test_handle_built_again_across_the_thread_line(O, sizes):
    graph = None
    for n in sizes:
        pb = envgen.geometric(5, d=3, n=n, nbox=5, r=0.2)
        pl = Planner(pb)
        if graph is not None:
            pl.graph = graph
        pl.build().plan()
        graph = pl.graph
        _, _, _, parent, cost, _ = oracle_run(O, pb)
        assert np.array_equal(pl.parent.cpu().numpy(), parent)
        assert np.array_equal(bits(pl.cost.cpu().numpy()), bits(cost))


@pytest.mark.parametrize("d, n, lam, blocks", [(2, 900, 0.0, 1), (2, 900, 0.2, 1), (2, 900, 0.5, -16), (2, 2048, 0.0, 1),
                                               (2, 2048, 0.2, -16), (2, 2049, 0.0, -16), (3, 900, 0.0, -16)])
def test_narrow_groups_of_small_2d_graphs_on_one_cta(O, d, n, lam, blocks):
    # their iterations hold a few nodes each: the cluster's barriers cost more than its warps give
    pb = envgen.geometric(5, d=d, n=n, nbox=5, r=0.12, lam=lam)
    pl = Planner(pb).build()
    info = pl.plan()
    assert N.gmt_graph_get_profile(pl.graph)["plan_blocks"] == blocks
    _, _, _, parent, cost, oinfo = oracle_run(O, pb)
    shared = N.gmt_graph_get_view(pl.graph)
    again = [torch.zeros_like(pl.parent), torch.zeros_like(pl.cost)]
    static = N.gmt_plan_static(pl.space, shared, pl.boxes, pl.params, again[0].data_ptr(), again[1].data_ptr(), None)
    for p, c, i in ((pl.parent, pl.cost, info), (*again, static.as_dict())):
        assert np.array_equal(p.cpu().numpy(), parent)
        assert np.array_equal(bits(c.cpu().numpy()), bits(cost))
        assert i["iters"] == oinfo["iters"] and i["checks"] == oinfo["checks"]
