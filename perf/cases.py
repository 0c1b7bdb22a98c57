"""The calls this planner's users make, at the sizes they make them: single plans (build and plan of one
problem), roadmap builds, batches of queries, the replanning server, and the learned proposal's forward pass,
training step and GEMM.

A case is a dict of plain values; `call` names what it does:
  plan     Planner.build(asynchronous=True) + Planner.plan(): a control loop's step on a new problem
  graph    Planner.build() + Planner.view(): samples and neighbour CSR, copied out by a program that keeps the roadmap
  batch    BatchPlanner.plan(): many uneven queries in one call
  serve    two ticks of the replanning server: every session's boxes have moved, every request is answered
  forward  Model.forward(): sampling logits of B environments
  train    Model.train_step(): loss, gradients and updated weights of one AdamW step
  gemm     gmt_gemm_bf16(): the tensor-core product the network is made of
"""
import math

import numpy as np
import torch

from paper_1705_02403_gb300 import _native as N
from paper_1705_02403_gb300 import envgen, learned, serving
from paper_1705_02403_gb300.planner import (BatchPlanner, Planner, goal_struct, params_struct, space_struct,
                                            wrap_device)

# Server shape of the replanning stream's own program (serving.run_stream's defaults).
SLOTS, CLUSTER, THREADS = 32, 4, 512


def listed():
    return [
        # The 2D workload of configs/geometric_2d_n1024.json: the smallest step there is, a launch-bound chain.
        {"name": "plan_2d_n1024", "call": "plan", "space": "geo", "d": 2, "n": 1024, "boxes": 10, "r": 0.12,
         "lam": 0.5},
        # The benchmark's workload, configs/double_integrator_6d_n4096.json.
        {"name": "plan_di_n4096", "call": "plan", "space": "di", "d": 6, "n": 4096, "boxes": 30, "lam": 0.5},
        # Dubins airplane in a forest of 1500 boxes, Halton samples and lambda = 1 as in the paper's Table 3.
        {"name": "plan_dubins_n5000_b1500", "call": "plan", "space": "dubins", "d": 4, "n": 5000, "boxes": 1500,
         "lam": 1.0},
        # 3D at the sample count of the learned proposal's solved training environments, one problem at a time.
        {"name": "plan_3d_n16384", "call": "plan", "space": "geo", "d": 3, "n": 16384, "boxes": 30, "r": 0.0,
         "lam": 0.5},
        # Table 1's "Rectangles" in 6D: a dense graph (thousands of neighbours a node), the sweeps' setting.
        {"name": "plan_rect6d_n5000", "call": "plan", "space": "rect", "d": 6, "n": 5000, "boxes": 10, "lam": 0.5},
        # A large 3D roadmap, built once and handed to the caller as CSR.
        {"name": "graph_3d_n65536", "call": "graph", "space": "geo", "d": 3, "n": 65536, "boxes": 30, "r": 0.0,
         "lam": 0.5},
        # 256 uneven 2D and 3D queries of 512 to 16384 samples: the batched benchmark.
        {"name": "batch_uneven_256", "call": "batch", "space": "uneven", "q": 256, "n_min": 512, "n_max": 16384},
        # 200 environments of the learned proposal's evaluation, planned together with uniform samples.
        {"name": "batch_env3d_200", "call": "batch", "space": "env3d", "q": 200, "n_min": 2048, "n_max": 2048},
        # The 100 Hz replanning stream: 100 double-integrator sessions whose 30 boxes move every tick.
        {"name": "serve_di_100", "call": "serve", "sessions": 100, "n_min": 2048, "n_max": 8192},
        # One environment's sampling logits: what stands before a single learned plan.
        {"name": "forward_b1", "call": "forward", "b": 1, "grid": 32, "hidden": 512, "cells": 16},
        # One training step at the training program's batch.
        {"name": "train_b256", "call": "train", "b": 256, "grid": 32, "hidden": 512, "cells": 16},
        # The GEMM entry point at the largest batch a model takes, with a bias: a square, compute-bound product.
        {"name": "gemm_4096", "call": "gemm", "m": 4096, "n": 4096, "k": 4096, "epilogue": 2},
    ]


def draw(rng):
    """One more case: sizes log-uniform over the listed ones' ranges, odd sizes among them."""
    def log(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    call = rng.choice(["plan", "plan", "plan", "graph", "batch", "serve", "forward", "train", "gemm"])
    if call in ("plan", "graph"):
        space = rng.choice(["geo2", "geo3", "di", "dubins", "rect"])
        lam = rng.choice([0.2, 0.5, 1.0])
        if space == "geo2":
            return {"call": call, "space": "geo", "d": 2, "n": log(256, 65536), "boxes": log(5, 80), "r": 0.0,
                    "lam": lam}
        if space == "geo3":
            return {"call": call, "space": "geo", "d": 3, "n": log(512, 49152), "boxes": log(5, 80), "r": 0.0,
                    "lam": lam}
        if space == "di":
            return {"call": call, "space": "di", "d": 6, "n": log(1024, 8192), "boxes": log(10, 300), "lam": lam}
        if space == "dubins":
            return {"call": call, "space": "dubins", "d": 4, "n": log(1000, 8000), "boxes": 10 * log(15, 500),
                    "lam": lam}
        return {"call": call, "space": "rect", "d": rng.randint(4, 10), "n": log(500, 5000), "boxes": 10, "lam": lam}
    if call == "batch":
        if rng.random() < 0.5:
            return {"call": call, "space": "uneven", "q": log(16, 200), "n_min": 512, "n_max": log(2048, 16384)}
        n = log(512, 4096)
        return {"call": call, "space": "env3d", "q": log(16, 200), "n_min": n, "n_max": n}
    if call == "serve":
        return {"call": call, "sessions": log(8, 80), "n_min": 2048, "n_max": log(2500, 8192)}
    if call == "forward":
        return {"call": call, "b": log(1, 256), "grid": rng.choice([16, 32]), "hidden": rng.choice([256, 512]),
                "cells": rng.choice([8, 16])}
    if call == "train":
        return {"call": call, "b": log(16, 256), "grid": rng.choice([16, 32]), "hidden": rng.choice([256, 512]),
                "cells": rng.choice([8, 16])}
    return {"call": call, "m": log(100, 4000), "n": log(100, 4000), "k": 8 * log(16, 500),
            "epilogue": rng.choice([0, 1, 2])}


# ---------------------------------------------------------------- inputs
def _problem(case, seed):
    s, n, lam = case["space"], case["n"], case["lam"]
    if s == "geo":
        return envgen.geometric(seed, d=case["d"], n=n, nbox=case["boxes"], r=case["r"], lam=lam)
    if s == "di":  # the frozen radius at 4096 samples, scaled to the same mean out-degree elsewhere
        return envgen.di6(seed, n=n, nbox=case["boxes"], r=serving.R_4096 * (4096.0 / n) ** (1.0 / 6.0), lam=lam)
    if s == "dubins":
        # the sampler draws the same Halton points for every seed; the seed places the trunks
        return envgen.dubins_forest(seed, n=n, trunks=10, strips=case["boxes"] // 10, lam=lam, sampler=1)
    return envgen.rectangles(seed, case["d"], n=n, nbox=case["boxes"], lam=lam)


def _queries(case, seed):
    """The seed places boxes and samples; how many samples and boxes each query has belongs to the case."""
    if case["space"] == "uneven":
        shapes = envgen.batch_queries(0, q=case["q"], n_min=case["n_min"], n_max=case["n_max"])
        return [envgen.geometric(seed * 1000 + k, d=pb.d, n=pb.n, nbox=pb.nbox, r=0.0, lam=pb.lam)
                for k, pb in enumerate(shapes)]
    return [learned.env(seed * 1000 + k, case["n_min"]) for k in range(case["q"])]


def _network_inputs(case, seed):
    """Voxel maps of 30 random boxes each, start and goal near opposite corners, and a target histogram along a
    bent line between them, as the training program's environments have them."""
    b, g, c = case["b"], case["grid"], case["cells"]
    rng = np.random.default_rng([seed, 7])
    side, mid = rng.uniform(0.05, 0.3, (2, b, 30, 3)), rng.uniform(0.0, 1.0, (2, b, 30, 3))
    lo = torch.from_numpy(mid[0] - side[0] / 2).float().cuda()
    hi = torch.from_numpy(mid[0] + side[0] / 2).float().cuda()
    p = (torch.arange(g, device="cuda") + 0.5) / g
    inside = ((lo[..., None] <= p) & (p <= hi[..., None])).float()  # [b, 30, 3, g]
    x = torch.einsum("bnx,bny,bnz->bxyz", inside[:, :, 0], inside[:, :, 1], inside[:, :, 2]) > 0
    x = x.reshape(b, g ** 3).to(torch.bfloat16).contiguous()
    start, goal = rng.uniform(0.02, 0.25, (b, 3)), rng.uniform(0.75, 0.98, (b, 3))
    sg = torch.from_numpy(np.concatenate([start, goal], 1)).float().cuda().contiguous()
    t = np.linspace(0.0, 1.0, 150)[None, :, None]
    bend = rng.uniform(-0.3, 0.3, (b, 1, 3))
    path = np.clip(start[:, None] * (1 - t) + goal[:, None] * t + bend * np.sin(np.pi * t), 0.0, 1.0 - 1e-6)
    cell = (path * c).astype(np.int64)
    cell = torch.from_numpy((cell[..., 0] * c + cell[..., 1]) * c + cell[..., 2]).cuda()
    target = torch.full((b, c ** 3), 1e-4, device="cuda")
    target.scatter_add_(1, cell, torch.ones_like(cell, dtype=torch.float32))
    return x, sg, (target / target.sum(1, keepdim=True)).contiguous()


def _model(case, seed):
    return N.Model(grid=case["grid"], hidden=case["hidden"], cells=case["cells"], max_batch=case["b"], seed=seed + 1)


def _gemm_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    a = torch.randn(case["m"], case["k"], generator=g, device="cuda").to(torch.bfloat16)
    b = torch.randn(case["n"], case["k"], generator=g, device="cuda").to(torch.bfloat16)
    return a, b, torch.randn(case["n"], generator=g, device="cuda")


class _Stream:
    """A server with its sessions open, and two ticks of their moving boxes."""

    def __init__(self, case, seed):
        rng = np.random.default_rng(9)  # the sessions' sizes belong to the case, their problems to the seed
        self.server = N.Server(slots=SLOTS, cluster=CLUSTER, threads=THREADS, max_nodes=case["n_max"] + 1,
                               max_boxes=30)
        self.sids, self.ticks, rows, total = [], [[], []], [], 0
        for k in range(case["sessions"]):
            n = int(rng.integers(case["n_min"], case["n_max"] + 1))
            pb = serving.session_problem(seed * 1000 + k, n)
            sid, _ = self.server.open_session(space_struct(pb), pb.x_init, goal_struct(pb), params_struct(pb),
                                              pb.box_lo, pb.box_hi)
            mover = serving.MovingBoxes(pb, seed * 1000 + k)
            for tick in self.ticks:
                tick.append(mover.step())
            self.sids.append(sid)
            rows.append(total)
            total += pb.N
        self.parent = torch.zeros(2, total, dtype=torch.int32, device="cuda")
        self.cost = torch.zeros(2, total, dtype=torch.float32, device="cuda")
        # each request as the loop sends it: session, request id, boxes, where its tree goes
        s = case["sessions"]
        self.requests = [[(self.sids[k], t * s + k, *self.ticks[t][k], self.parent[t].data_ptr() + 4 * rows[k],
                           self.cost[t].data_ptr() + 4 * rows[k]) for k in range(s)] for t in range(2)]

    def run(self):
        s = len(self.sids)
        goal, path_cost, checks = np.zeros(2 * s, np.int32), np.zeros(2 * s, np.float32), np.zeros(2 * s, np.int64)
        edges, status = np.zeros(2 * s, np.int64), np.zeros(2 * s, np.int32)
        for requests in self.requests:
            for request in requests:
                self.server.submit(*request)
            done = 0
            while done < s:
                for r in self.server.poll(s, 100):
                    i = r["request_id"]
                    goal[i], path_cost[i], checks[i] = r["goal_node"], r["path_cost"], r["checks"]
                    edges[i], status[i] = r["edges_checked"], r["status"]
                    done += 1
        return {"parent": self.parent, "cost": self.cost, "status": status, "goal_node": goal,
                "path_cost": path_cost, "checks": checks, "edges_checked": edges}


def prepare(case, seed):
    call = case["call"]
    if call in ("plan", "graph"):
        pl = Planner(_problem(case, seed))
        pl.path.zero_()  # a plan writes the path's own entries only
        if call == "plan":
            return {"call": call, "planner": pl}
        # the program's own roadmap, with room for any seed's edges
        room = _edge_room(case)
        names = ("out", "in") if case["space"] in ("di", "dubins") else ("out",)
        return {"call": call, "planner": pl,
                "col": {k: torch.zeros(room, dtype=torch.int32, device="cuda") for k in names},
                "cost": {k: torch.zeros(room, dtype=torch.float32, device="cuda") for k in names}}
    if call == "batch":
        return {"call": call, "planner": BatchPlanner(_queries(case, seed))}
    if call == "serve":
        return {"call": call, "stream": _Stream(case, seed)}
    if call == "gemm":
        a, b, bias = _gemm_inputs(case, seed)
        return {"call": call, "a": a, "b": b, "bias": bias, "epilogue": case["epilogue"]}
    x, sg, target = _network_inputs(case, seed)
    m = _model(case, seed)
    state = {"call": call, "model": m, "b": case["b"], "x": x, "sg": sg, "target": target}
    if call == "forward":
        state["logits"] = torch.zeros(case["b"], case["cells"] ** 3, device="cuda")
        return state
    v = m.view()
    h, d, z, c = v.hidden, v.in_features, v.z_features, v.n_cells
    shapes = {"W1": (h, d), "b1": (h,), "W2": (h, h), "b2": (h,), "W3": (c, z), "b3": (c,)}
    state["out"] = {name: wrap_device(getattr(v, name), shape, "f4", m) for name, shape in shapes.items()}
    state["out"] |= {"g" + name: wrap_device(getattr(v, "g" + name), shape, "f4", m)
                     for name, shape in shapes.items()}
    state["out"]["logits"] = wrap_device(v.logits, (case["b"], c), "f4", m)
    return state


# ---------------------------------------------------------------- one pass
def run(state):
    call = state["call"]
    if call == "plan":
        pl = state["planner"]
        pl.build(asynchronous=True)
        info = pl.plan()
        return {"parent": pl.parent, "cost": pl.cost, "path": pl.path, "info": info}
    if call == "graph":
        v = state["planner"].build().view()
        for k, to in state["col"].items():  # a Euclidean graph's in-edges are its out-edges
            to[:v.E].copy_(getattr(v, k + "_col"))
            state["cost"][k][:v.E].copy_(getattr(v, k + "_cost"))
        return {"X": v.X, "is_goal": v.is_goal, "out_row": v.out_row, "in_row": v.in_row, "col": state["col"],
                "cost": state["cost"]}
    if call == "batch":
        bp = state["planner"]
        infos = np.frombuffer(bp.plan(raw=True), dtype=np.dtype(N.gmt_plan_info))
        return {"parent": bp.parent, "cost": bp.cost, "info": {f: infos[f] for f in infos.dtype.names}}
    if call == "serve":
        return state["stream"].run()
    if call == "gemm":
        out, error = N.gmt_gemm_bf16(state["a"], state["b"], epilogue=state["epilogue"],
                                     bias=state["bias"] if state["epilogue"] else None)
        return {"c": out, "error": error}
    m, b = state["model"], state["b"]
    if call == "forward":
        m.forward(b, state["x"].data_ptr(), state["sg"].data_ptr(), state["logits"].data_ptr())
        return {"logits": state["logits"]}
    # the training program's learning rate and weight decay
    loss = m.train_step(b, state["x"].data_ptr(), state["sg"].data_ptr(), state["target"].data_ptr(), 1e-3, 1e-4)
    return {"loss": loss, **state["out"]}


# ---------------------------------------------------------------- work
def _degree(case, n):
    """About how many neighbours a node has (each edge once per direction)."""
    if case["space"] == "di":
        return 40.0  # what the frozen radius was chosen for
    if case["space"] == "dubins":
        return 14.0 * n / 5000.0
    d = case.get("d", 3)
    zeta = math.pi ** (d / 2) / math.gamma(d / 2 + 1)
    r = case.get("r") or 4.0 * ((1.0 / d) / zeta * math.log(n) / n) ** (1.0 / d)
    return min(n / 2.0, n * zeta * r ** d)


def _edge_room(case):
    """More edges than a graph of the case has: boxes crowd the samples, in 2D to several times the density."""
    n = case["n"] + 1
    return int(min(float(n) * n, (6.0 if case["d"] == 2 else 2.5) * n * _degree(case, n)))


def _plan_work(case, n):
    """One build and plan: the boxes read and the outputs written once, every edge (column and cost) written once
    and read once, and about 30 operations an edge (its cost, and its part in a minimum)."""
    e = n * _degree(case, n)
    return {"bytes": 16.0 * e + n * (4.0 * case.get("d", 3) + 8.0) + 32.0 * case.get("boxes", 30), "flops": 30.0 * e}


def work(case):
    call = case["call"]
    if call == "plan":
        return _plan_work(case, case["n"])
    if call == "graph":
        e = case["n"] * _degree(case, case["n"])
        directed = 2.0 if case["space"] in ("di", "dubins") else 1.0
        return {"bytes": 8.0 * e * directed + case["n"] * (4.0 * case["d"] + 9.0), "flops": 10.0 * e}
    if call in ("batch", "serve"):
        # log-uniform sizes' mean; two ticks replan on a graph that is there: its edges read once each
        lo, hi = case["n_min"], case["n_max"]
        n = (hi - lo) / math.log(hi / lo) if call == "batch" and hi > lo else (lo + hi) / 2.0
        count = case["q"] if call == "batch" else 2 * case["sessions"]
        one = _plan_work({"space": "di", "d": 6} if call == "serve" else {"space": "geo", "d": 3}, n)
        return {k: v * count * (0.5 if call == "serve" and k == "bytes" else 1.0) for k, v in one.items()}
    if call == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 2.0 * (m + n) * k + (2.0 if case["epilogue"] == 1 else 4.0) * m * n, "flops": 2.0 * m * n * k}
    b, g, h, c = case["b"], case["grid"] ** 3, case["hidden"], case["cells"] ** 3
    weights = h * g + h * h + c * (h + 16)
    if call == "forward":
        return {"bytes": 2.0 * weights + 2.0 * b * g + 4.0 * b * c, "flops": 2.0 * b * weights}
    # weights read as BF16, then master weight, both moments read and written, gradient and BF16 copy written;
    # three products, less the input's gradient
    return {"bytes": 32.0 * weights + 2.0 * b * g + 8.0 * b * c, "flops": 2.0 * b * (3.0 * weights - h * g)}


# ---------------------------------------------------------------- in 64 bits
def _philox(c, key):
    """Philox4x32-10 of counters c (four int64 tensors of 32-bit values)."""
    mask = 0xFFFFFFFF

    def mul(x, m):  # high and low words of a 32 x 32 bit product
        lo, hi = x * (m & 0xFFFF), x * (m >> 16)
        return (hi + (lo >> 16)) >> 16, (((hi & 0xFFFF) << 16) + lo) & mask

    k0, k1 = key & mask, (key >> 32) & mask
    for _ in range(10):
        ha, la = mul(c[0], 0xD2511F53)
        hb, lb = mul(c[2], 0xCD9E8D57)
        c = [hb ^ c[1] ^ k0, lb, ha ^ c[3] ^ k1, la]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _exact_samples(pb):
    """SampleFree: node k keeps the first of its attempts outside every box (node 1: inside the goal ball too)."""
    dev = "cuda"
    lo, hi = (torch.from_numpy(v).to(dev) for v in (pb.box_lo, pb.box_hi))
    x = torch.zeros(pb.N, pb.d, device=dev)
    x[0] = torch.from_numpy(pb.x_init).to(dev)
    centre = torch.from_numpy(pb.goal_center).to(dev)
    todo = torch.arange(1, pb.N, device=dev)
    t = 0
    while todo.numel():
        zero = torch.zeros_like(todo)
        w = _philox([todo, zero + t, zero, zero], pb.seed)
        u = torch.stack([(v >> 8).float() * 2.0 ** -24 for v in w[:pb.d]], 1)
        slo, shi = (torch.from_numpy(v).to(dev).expand(todo.numel(), pb.d).clone() for v in (pb.lo, pb.hi))
        first = todo == 1
        rho = np.float32(pb.goal_radius)
        slo[first], shi[first] = centre - float(rho), centre + float(rho)
        p = slo + u * (shi - slo)
        hit = ((lo <= p[:, None]) & (p[:, None] <= hi)).all(2).any(1)
        d2 = torch.zeros_like(p[:, 0])
        for a in range(pb.d):
            d2 = d2 + (p[:, a] - centre[a]) * (p[:, a] - centre[a])
        ok = ~hit & (~first | ((d2 <= float(rho * rho)) & (p >= 0).all(1) & (p <= 1).all(1)))
        x[todo[ok]] = p[ok]
        todo = todo[~ok]
        t += 1
    return x


def _exact_graph(case, seed):
    """Samples, and the cost in 64 bits of every pair that the FP32 distance says is nearer than r."""
    if case["space"] not in ("geo", "rect") or case["d"] > 4:
        # DI and Dubins: which pairs are edges is decided in rounded arithmetic that 64 bits do not share;
        # over four axes the distance's rounding decides pairs too often to lay the edges out the same
        return None
    pb = _problem(case, seed)
    d, n = pb.d, pb.n
    r = pb.r
    if r <= 0.0:
        zeta = math.pi ** (d / 2) / math.gamma(d / 2 + 1)
        r = 4.0 * ((1.0 / d) / zeta * math.log(n) / n) ** (1.0 / d)
    r = float(np.float32(r))
    x = _exact_samples(pb)
    costs = []
    step = max(1, (1 << 26) // pb.N)
    for i in range(0, pb.N, step):
        s = torch.zeros(min(step, pb.N - i), pb.N, device=x.device)
        for a in range(d):
            t = x[None, :, a] - x[i:i + step, a, None]
            s = s + t * t
        near = s.sqrt() < r
        near[torch.arange(near.shape[0]), torch.arange(i, i + near.shape[0])] = False
        row, col = near.nonzero(as_tuple=True)
        costs.append((x[row + i].double() - x[col].double()).square().sum(1).sqrt())
    costs = torch.cat(costs)
    cost = torch.zeros(_edge_room(case), dtype=torch.float64, device=x.device)
    cost[:costs.numel()] = costs
    return {"X": x.double().T.contiguous(), "is_goal": None, "out_row": None, "in_row": None, "col": None,
            "cost": {"out": cost}}


def _exact_network(case, seed):
    x, sg, target = (v.double() for v in _network_inputs(case, seed))
    b, h, c = case["b"], case["hidden"], case["cells"] ** 3
    d, z = case["grid"] ** 3, h + 16
    w = []
    for i, (rows, cols, var) in enumerate(((h, d, 2.0 / d), (h, h, 2.0 / h), (c, z, 1.0 / z))):
        t = torch.arange(rows * cols, device=x.device)
        zero = torch.zeros_like(t)
        u = _philox([t, zero, zero + 3, zero + i], seed + 1)
        normal = torch.sqrt(-2.0 * torch.log(((u[0] >> 8) + 1).double() * 2.0 ** -24)) * \
            torch.cos(2.0 * math.pi * (u[1] >> 8).double() * 2.0 ** -24)
        # the products read the weights' BF16 copies
        w.append((math.sqrt(var) * normal).float().to(torch.bfloat16).double().reshape(rows, cols))
        del u, normal, t, zero
    h1 = (x @ w[0].T).relu()
    h2 = (h1 @ w[1].T).relu()
    zz = torch.cat([h2, sg, torch.zeros(b, z - h - 6, dtype=torch.float64, device=x.device)], 1)
    logits = zz @ w[2].T
    if case["call"] == "forward":
        return {"logits": logits}
    logp = torch.log_softmax(logits, 1)
    dl = (logp.exp() - target) / b
    dh2 = (dl @ w[2])[:, :h] * (h2 > 0)
    dh1 = (dh2 @ w[1]) * (h1 > 0)
    # AdamW's first step divides a gradient by its own magnitude, so the updated weights have no value of their own
    # where that gradient is rounding noise
    return {"loss": float(-(target * logp).sum(1).mean()), "gW1": dh1.T @ x, "gb1": dh1.sum(0), "gW2": dh2.T @ h1,
            "gb2": dh2.sum(0), "gW3": dl.T @ zz, "gb3": dl.sum(0), "logits": logits, "W1": None, "b1": None,
            "W2": None, "b2": None, "W3": None, "b3": None}


def exact(case, seed):
    call = case["call"]
    if call == "graph":
        return _exact_graph(case, seed)
    if call == "gemm":
        a, b, bias = (v.double() for v in _gemm_inputs(case, seed))
        c = a @ b.T
        if case["epilogue"]:
            c = c + bias
        return {"c": c.relu() if case["epilogue"] == 1 else c, "error": None}
    if call in ("forward", "train"):
        return _exact_network(case, seed)
    # A tree's costs follow from which node joined in which group under FP32 thresholds and collision tests; the same
    # algorithm in 64 bits grows another tree, so a planned cost has no 64-bit value of its own.
    return None
