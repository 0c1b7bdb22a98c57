"""Several host threads, a handle each: calls whose kernels need different
amounts of shared memory, at the same time.  Every call succeeds and leaves the
bits of the same call alone (one handle in two calls at once is the only
sharing the API forbids)."""
import threading

import numpy as np
import pytest
import torch

from paper_1705_02403_gb300 import _native as N
from paper_1705_02403_gb300 import envgen
from paper_1705_02403_gb300.planner import BatchPlanner, Planner, goal_struct, params_struct, space_struct

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def together(jobs, passes):
    """jobs: (call of a stream, its outputs); each call runs `passes` times on its own thread and stream."""
    alone = []
    for call, outputs in jobs:
        call(None)
        alone.append(outputs())
    errors, last = [], [None] * len(jobs)
    start = threading.Barrier(len(jobs))

    def loop(k):
        stream = torch.cuda.Stream().cuda_stream
        start.wait()
        for _ in range(passes):
            try:
                jobs[k][0](stream)
            except N.GmtError as e:
                errors.append(str(e))
        last[k] = jobs[k][1]()
    threads = [threading.Thread(target=loop, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, f"{len(errors)} of {passes * len(jobs)} calls: {errors[0]}"
    for got, want in zip(last, alone):
        assert all(np.array_equal(g, w) for g, w in zip(got, want))


def words(*tensors):
    return [t.cpu().numpy().view(np.int32) for t in tensors]


def planned(pb):
    pl = Planner(pb).build()
    return pl.plan, lambda: words(pl.parent, pl.cost)


def built(pb):
    pl = Planner(pb)

    def rows():
        v = pl.view()
        return words(v.out_row, v.out_col, v.out_cost)
    return pl.build, rows


def batched(pbs):
    kept = []

    def call(stream):  # a batch of its own each time: first passes set more limits than replays
        kept[:] = [BatchPlanner(pbs)]
        kept[0].plan(stream)
    return call, lambda: words(kept[0].parent, kept[0].cost)


def geo(seed, n):
    return envgen.geometric(seed, d=2, n=n, nbox=4, r=0.2)


def test_plans_of_different_sizes():
    together([planned(geo(k, 60 if k % 2 else 1500)) for k in range(12)], 2000)


def test_double_integrator_plans_of_different_sizes():
    together([planned(envgen.di6(seed=k, n=300 if k % 2 else 4096, r=2.6)) for k in range(6)], 800)


def test_cell_builds_of_different_sizes():
    together([built(envgen.geometric(k, d=3, n=20000 if k % 2 else 70000, nbox=5, r=0.04)) for k in range(4)], 150)


def test_batches_of_different_sizes():
    together([batched([geo(i, 200 if k % 2 else 3000) for i in range(3)]) for k in range(4)], 60)


def test_plans_beside_a_server():
    sessions = [envgen.di6(seed=5 + k, n=n, r=2.6) for k, n in enumerate((2048, 3000, 8192))]
    server = N.Server(slots=3, cluster=4, threads=512, max_nodes=8193, max_boxes=30)
    sids = [server.open_session(space_struct(p), p.x_init, goal_struct(p), params_struct(p), p.box_lo, p.box_hi)[0]
            for p in sessions]
    out = [(torch.zeros(p.N, dtype=torch.int32, device="cuda"), torch.zeros(p.N, device="cuda")) for p in sessions]

    def serve(stream):
        for k, (sid, p) in enumerate(zip(sids, sessions)):
            server.submit(sid, k, p.box_lo, p.box_hi, out[k][0].data_ptr(), out[k][1].data_ptr())
        results = []
        while len(results) < len(sids):
            results += server.poll(16, 100)
        for r in results:
            if r["status"] < 0:
                raise N.GmtError(r["status"], "a served request")
    together([planned(envgen.di6(seed=4, n=n, r=2.428)) for n in (300, 4096, 300, 4096)] +
             [(serve, lambda: words(*(v for pair in out for v in pair)))], 500)
    server.close()
