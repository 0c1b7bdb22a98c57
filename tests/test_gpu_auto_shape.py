"""The automatic launch shape of a handle that is built again at another size:
it is chosen for the graph the handle holds now, and the tree is the oracle's."""
import numpy as np
import pytest
import torch

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
