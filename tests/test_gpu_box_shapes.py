"""Box grids of uneven obstacles: walls across the domain, a few boxes many
times larger than the rest, slices along either axis, boxes without a point and
boxes beyond the domain.  Trees equal the oracle's bit for bit, whatever shape
the grid takes; and a few large boxes do not make every point test them all."""
import time

import numpy as np
import pytest
import torch

from paper_1705_02403_gb300 import envgen
from paper_1705_02403_gb300.planner import Planner
from test_gpu_parity import assert_same, gpu_run, oracle_run

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module")
def P():
    from paper_1705_02403_gb300 import planner
    return planner


def with_boxes(pb, kind, count, density=0.15):
    rng = np.random.default_rng([count, pb.dp])
    c = rng.uniform(0.12, 0.88, (count, pb.dp))
    s = np.full((count, pb.dp), (density / count) ** (1.0 / pb.dp))
    if kind == "mixed":  # alternating slices along the first and the second axis
        s[::2, 0] *= 4
        s[::2, 1] /= 4
        s[1::2, 0] /= 4
        s[1::2, 1] *= 4
    elif kind == "wide":
        s[:, 0] *= 16
        s[:, 1] /= 16
    elif kind == "tall":
        s[:, 1] *= 16
        s[:, 0] /= 16
    elif kind == "skew":
        s[:count // 10] *= 4
    elif kind == "walls":  # eight thin ones, three quarters of the domain long
        s[:8] = 0.004
        s[:4, 0], c[:4, 0] = 0.75, 0.625
        s[4:8, 1], c[4:8, 1] = 0.75, 0.375
    elif kind == "odd":
        s[:5] = -s[:5]             # no point
        s[5, 1], c[5, 1] = 0.5, 1.3  # in part beyond the domain
        c[6] = 3.0                 # beyond it
        s[7:20] = 0.0              # a point each
    lo, hi = c - s / 2, c + s / 2  # none over the start or the goal
    near = (lo < 0.12).all(1) & (hi > 0.0).all(1) | (hi > 0.88).all(1) & (lo < 1.0).all(1)
    c[near], s[near] = 0.5, 0.001
    pb.box_lo, pb.box_hi = (c - s / 2).astype(np.float32), (c + s / 2).astype(np.float32)
    return pb


@pytest.mark.parametrize("count", [128, 1025, 5000, 8192])
@pytest.mark.parametrize("kind", ["mixed", "wide", "tall", "skew", "walls", "odd"])
@pytest.mark.parametrize("d", [2, 3])
def test_uneven_boxes(O, P, d, kind, count):
    pb = with_boxes(envgen.geometric(count, d=d, n=250, nbox=0, r=0.2 if d == 2 else 0.3), kind, count)
    assert_same(O, gpu_run(P, pb), *oracle_run(O, pb))


def test_a_few_large_boxes_are_not_tested_everywhere():
    def best(kind):
        pl = Planner(with_boxes(envgen.geometric(3, d=2, n=1000, nbox=0, r=0.12), kind, 1500))
        t = []
        for _ in range(30):
            t0 = time.perf_counter()
            pl.build(asynchronous=True).plan()
            t.append(time.perf_counter() - t0)
        return min(t)
    # a tenth of the boxes four times wider: two and a half times the area, against 5.5 times the time
    # when they went over too many cells to be listed
    assert best("skew") < 3.0 * best("even")


def test_lists_of_many_boxes_are_not_written_by_one_block():
    def best(count):
        rng = np.random.default_rng(count)
        pb = envgen.di6(seed=3, n=1000, nbox=1, r=2.7)
        c, side = rng.uniform(0.12, 0.88, (count, 3)), (0.15 / count) ** (1 / 3)
        pb.box_lo, pb.box_hi = (c - side / 2).astype(np.float32), (c + side / 2).astype(np.float32)
        pl = Planner(pb)
        t = []
        for _ in range(30):
            t0 = time.perf_counter()
            pl.build(asynchronous=True).plan()
            t.append(time.perf_counter() - t0)
        return min(t)
    # 1.8 times the time of as many boxes again when one block wrote every list
    assert best(8190) < 1.6 * best(8200)


@pytest.mark.parametrize("count", [255, 256, 257, 300])
@pytest.mark.parametrize("d", [2, 3, 4])
def test_counts_around_the_scatter_line(O, P, d, count):
    pb = with_boxes(envgen.geometric(count, d=d, n=250, nbox=0, r=0.3 if d < 4 else 0.6), "mixed", count)
    assert_same(O, gpu_run(P, pb), *oracle_run(O, pb))
