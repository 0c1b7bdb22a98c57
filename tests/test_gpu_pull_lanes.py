"""Batched pulls by half warps or whole warps: iterations on both sides of the
rule's line give the trees and counters of the single plan."""
import numpy as np
import pytest
import torch

from paper_1705_02403_gb300 import _native as N
from paper_1705_02403_gb300 import envgen
from paper_1705_02403_gb300.planner import BatchPlanner, Planner

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

KEYS = ("status", "goal_node", "path_len", "iters", "final_i", "push_edges", "pull_edges", "checks", "failed", "tree_size")


def problems(kind):
    if kind == "di":
        return [envgen.di6(40 + k, n=600 + 150 * k, r=2.8) for k in range(3)]
    d = 2 if kind == "2d" else 3
    # a wide radius opens most nodes in one iteration, a narrow one a few at a time
    return [envgen.geometric(60 + k, d=d, n=n, nbox=6, r=r, lam=lam)
            for k, (n, r, lam) in enumerate([(1500, 0.6, 1.0), (1500, 0.2, 0.3), (40, 0.4, 0.5), (1500, 2.0, 1.0)])]


# 128 threads: 64 candidates of a CTA reach the line; 1024: 512 do
@pytest.mark.parametrize("cluster, threads", [(1, 128), (1, 256), (2, 128), (2, 1024), (4, 128)])
@pytest.mark.parametrize("kind", ["2d", "3d", "di"])
def test_pulls_match_single_plans(kind, cluster, threads):
    pbs = problems(kind)
    bp = BatchPlanner(pbs)
    bp.plan(allow_errors=True)
    N.gmt_batch_set_mode(bp.batch, N.BATCH_TEAMS)
    N.gmt_batch_set_launch(bp.batch, cluster, threads)
    infos = bp.plan(allow_errors=True)
    for k, pb in enumerate(pbs):
        pl = Planner(pb).build()
        want = pl.plan(allow_errors=True)
        assert [infos[k][f] for f in KEYS] == [want[f] for f in KEYS]
        parent, cost = bp.result(k)
        assert torch.equal(parent, pl.parent)
        assert np.array_equal(cost.cpu().numpy().view(np.int32), pl.cost.cpu().numpy().view(np.int32))
