"""A request whose launch the driver refuses (the regions of more than 1024
boxes that moved at once do not fit the invalidation's shared memory) leaves
its session as it was: the next request's tree is the oracle's, although edges
were checked before against boxes that have moved since."""
import numpy as np
import pytest
import torch

from paper_1705_02403_gb300 import _native as N
from paper_1705_02403_gb300 import envgen
from test_gpu_serving import assert_oracle, oracle_graph, structs

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("slots", [1, 2])
def test_next_request_after_a_refused_launch(O, slots):
    pb = envgen.geometric(11, d=3, n=800, nbox=0, r=0.3)
    rng = np.random.default_rng(5)
    large = 100
    mid = rng.uniform(0.15, 0.85, (1100, 3))
    half = np.where(np.arange(1100) < large, 0.04, 0.002)[:, None]
    to = mid.copy()
    to[:large] = rng.uniform(0.15, 0.85, (large, 3))  # the large boxes go elsewhere,
    to[large:] += 0.01                                # the small ones a step aside
    part = np.where(np.arange(1100)[:, None] < large, to, mid)

    def boxes(c):
        return (c - half).astype(np.float32), (c + half).astype(np.float32)
    pb.box_lo, pb.box_hi = boxes(mid)
    server = N.Server(slots=slots, cluster=2, threads=256, max_nodes=pb.N, max_boxes=1100)
    space, goal, params = structs(pb)
    sid, _ = server.open_session(space, pb.x_init, goal, params, pb.box_lo, pb.box_hi)
    parent = torch.zeros(pb.N, dtype=torch.int32, device="cuda")
    cost = torch.zeros(pb.N, device="cuda")
    g = oracle_graph(O, pb)

    def ask(c):
        server.submit(sid, 1, *boxes(c), parent.data_ptr(), cost.data_ptr())
        r = []
        while not r:
            r = server.poll(1, 100)
        return r[0]
    for c in (mid, to, part, mid):
        r = ask(c)
        if c is to:
            assert r["status"] == N.GMT_ERR_CUDA
        else:
            assert_oracle(O, g, pb, *boxes(c), r, parent, cost)
    server.close()
