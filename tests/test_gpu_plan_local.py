"""The wavefront with its state in the team's shared memory, at the sizes where
its node ownership, row parts and box grid change: node counts around multiples
of the team's CTAs and of 32 own nodes, rows around the length from which they
are read four entries at a time, iteration counts past the mark stamps' period,
box counts around the grid's limits, and graphs that take the other body.
Everything must equal the oracle bit for bit."""
import numpy as np
import pytest
import torch

from paper_1705_02403_gb300 import envgen
from test_gpu_parity import assert_same, gpu_run, oracle_run

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module")
def P():
    from paper_1705_02403_gb300 import planner
    return planner


@pytest.mark.parametrize("cluster", [1, 2, 3, 7, 16])
def test_node_counts_around_the_ownership_steps(O, P, cluster):
    launch = (1, 64) if cluster == 1 else (0, 64, cluster)
    for N in sorted({2, cluster, cluster + 1, 2 * cluster + 1, 32 * cluster - 1, 32 * cluster, 32 * cluster + 1}):
        if N < 2:
            continue
        pb = envgen.geometric(N, d=2, n=N - 1, nbox=3, r=0.3)
        assert_same(O, gpu_run(P, pb, launch=launch), *oracle_run(O, pb))


@pytest.mark.parametrize("n", [126, 127, 128, 129, 130, 131, 257, 258, 1100])
def test_complete_graphs_around_the_long_row_length(O, P, n):
    # every node a neighbour of every other: rows of n entries at every alignment
    pb = envgen.geometric(n, d=3, n=n, nbox=4, r=1.8)
    for launch in ((0, 128, 4), (0, 0)):
        assert_same(O, gpu_run(P, pb, launch=launch), *oracle_run(O, pb))


def test_more_iterations_than_mark_stamps(O, P):
    # lambda = 0: one iteration per distinct cost, several times the stamps' period of 255
    pb = envgen.geometric(9, d=2, n=900, nbox=8, r=0.1, lam=0.0)
    G = gpu_run(P, pb, launch=(0, 256, 8))
    assert G["info"]["iters"] > 600
    assert_same(O, G, *oracle_run(O, pb))


@pytest.mark.parametrize("count", [127, 128, 1024, 8192, 8193])
@pytest.mark.parametrize("d", [2, 3, 4])
def test_box_counts_around_the_grid_limits(O, P, d, count):
    rng = np.random.default_rng([count, d])
    pb = envgen.geometric(5, d=d, n=400, nbox=0, r={2: 0.15, 3: 0.35, 4: 0.5}[d])
    side = 0.4 / count ** (1.0 / d)
    lo, hi = envgen.random_boxes(rng, count, d, pb.x_init, pb.goal_center, 0.05, side=(0.1 * side, side))
    pb = pb.with_(box_lo=lo, box_hi=hi)
    assert_same(O, gpu_run(P, pb), *oracle_run(O, pb))


def test_rows_that_are_not_aligned(O, P):
    # caller arrays off the 16-byte boundary cannot be read four entries at a time
    from paper_1705_02403_gb300 import _native as N
    pb = envgen.geometric(3, d=3, n=500, nbox=6, r=0.5)
    X, goal, g, parent, cost, info = oracle_run(O, pb)
    pl = P.Planner(pb).build()
    v = pl.view()
    raw = v.raw

    def shifted(t):
        room = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")
        room[1:].copy_(t)
        return room
    keep = {k: shifted(getattr(v, k)) for k in ("out_col", "in_col", "in_cost")}
    for k, t in keep.items():
        setattr(raw, k, t.data_ptr() + 4)
    N.gmt_plan_static(pl.space, raw, pl.boxes, pl.params, pl.parent.data_ptr(), pl.cost.data_ptr())
    assert np.array_equal(pl.parent.cpu().numpy(), parent)
    assert np.array_equal(pl.cost.cpu().numpy().view(np.uint32), cost.view(np.uint32))


@pytest.mark.parametrize("q", [1, 9, 10, 38, 39, 100])
@pytest.mark.parametrize("big", [0, 21000, 120000])
def test_batches_at_the_untuned_shapes_limits(O, P, q, big):
    # teams from 16 CTAs (one query) to 2; a largest query whose state needs
    # more CTAs, and one whose state fits no team (scratch in global memory)
    if big and q not in (1, 39):
        pytest.skip("the largest query decides")
    qs = [envgen.geometric(700 + k, d=2 + k % 2, n=3 + 37 * (k % 11), nbox=5, r=0.35) for k in range(q)]
    if big:
        qs.append(envgen.geometric(9, d=2, n=big, nbox=12, r=0.012 if big < 50000 else 0.005))
    bp = P.BatchPlanner(qs)
    infos = bp.plan()
    for k in range(0, len(qs), 5):
        if qs[k].n > 1000:
            continue
        X, goal, g, parent, cost, info = oracle_run(O, qs[k])
        got_parent, got_cost = bp.result(k)
        assert np.array_equal(got_parent.cpu().numpy(), parent)
        assert np.array_equal(got_cost.cpu().numpy().view(np.uint32), cost.view(np.uint32))
        assert infos[k]["checks"] == info["checks"] and infos[k]["iters"] == info["iters"]
    if big:  # as planned alone
        pl = P.Planner(qs[-1]).build()
        info = pl.plan()
        got_parent, got_cost = bp.result(len(qs) - 1)
        assert torch.equal(got_parent, pl.parent) and torch.equal(got_cost.view(torch.int32), pl.cost.view(torch.int32))
        assert all(infos[-1][f] == info[f] for f in ("iters", "checks", "push_edges", "pull_edges", "goal_node"))
