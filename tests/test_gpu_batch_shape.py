"""The untuned shape of a batch's plan stage: as many threads as pay, by the
number of queries and their size; and the trees are those of another shape."""
import numpy as np
import pytest
import torch

from paper_1705_02403_gb300 import _native as N
from paper_1705_02403_gb300 import envgen
from paper_1705_02403_gb300.planner import BatchPlanner

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("q, n, cluster, threads", [(40, 1000, 2, 1024), (76, 200, 2, 1024), (77, 1000, 2, 256),
                                                    (40, 128, 2, 256), (30, 1000, 4, 512), (12, 1000, 8, 256),
                                                    (40, 1025, 2, 1024)])
def test_untuned_shape(q, n, cluster, threads):
    pbs = [envgen.dubins_forest(k, n=n, r=0.25, trunks=2, strips=10) if k % 2 else
           envgen.geometric(k, d=3, n=n, nbox=8, r=0.2) for k in range(q)]
    bp = BatchPlanner(pbs)
    infos = bp.plan()
    assert N.gmt_batch_get_launch(bp.batch)[1:] == (cluster, threads)
    want = [bp.parent.cpu().numpy(), bp.cost.cpu().numpy().view(np.int32)]
    N.gmt_batch_set_launch(bp.batch, 4, 256)
    again = bp.plan()
    assert np.array_equal(bp.parent.cpu().numpy(), want[0])
    assert np.array_equal(bp.cost.cpu().numpy().view(np.int32), want[1])
    assert [(i["iters"], i["checks"]) for i in again] == [(i["iters"], i["checks"]) for i in infos]
