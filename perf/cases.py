"""Workloads whose speed this project watches, each through the calls a user makes.

Every case is a dict of plain values; ``listed()`` gives the standing ones,
``draw(rng)`` another of the same ranges.  ``prepare`` makes what a program has
in hand (inputs on the device, a handle, weights), ``run`` is one pass and
returns its whole results, ``work`` the bytes and operations no implementation
can do without, and ``exact`` the same results in 64 bits by plain torch.

The kinds:

  schedule  Batched-Extension: from an empty graph, insert a block of vertices
            and edges and exploit to a stable policy, block after block; then
            read costs and parents.  Options: box dimension, block size, cost
            type, blocks resident on the device or copied from page-locked host
            memory while the previous block is exploited, and a goal.
  policy    one roadmap, a breadth-first initial policy handed in, one exploit.
  batch     many independent roadmaps merged and exploited in one launch.
  evaluate  costs-to-come of a given policy without any allocation.
  roadmap   k-nearest neighbours and collision-checked edges of given samples.
  forward / sample / train   the learned sampling proposal.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2003_04920_gb300 as pkg
from paper_2003_04920_gb300 import workloads as W
from paper_2003_04920_gb300.workloads import gpu as GG

PI = math.pi


def listed():
    return [
        # the smallest planning call: the oracle-sized 2-D r-disc scale with FP64
        # costs and an initial policy, a few hundred microseconds of launches
        dict(name="policy_2d_2k_f64", kind="policy", n=2001, dim=2, k=30, f64=True),
        # a planner that replans after every 100 samples of a small 2-D query
        # (the paper's block-size sweep at N = 10^4): latency per block
        dict(name="query_2d_10k_s100", kind="schedule", n=10_000, dim=2, k=51, block=100,
             f64=False, host=False, goal=True),
        # an ordinary 2-D roadmap in blocks of 10^4: deep trees
        dict(name="blocks_2d_200k", kind="schedule", n=200_000, dim=2, k=67, block=10_000,
             f64=False, host=False, goal=False),
        # an ordinary 6-D roadmap whose blocks arrive from page-locked host
        # memory, copied while the previous block is exploited; odd sizes
        dict(name="blocks_6d_500k_host", kind="schedule", n=500_003, dim=6, k=30, block=49_999,
             f64=False, host=True, goal=False),
        # the same toward a goal with an admissible heuristic
        dict(name="goal_6d_1m", kind="schedule", n=1_000_000, dim=6, k=30, block=50_000,
             f64=False, host=False, goal=True),
        # the headline benchmark: 4M vertices in 6-D, 80 blocks of 5*10^4
        dict(name="blocks_6d_4m", kind="schedule", n=4_000_000, dim=6, k=30, block=50_000,
             f64=False, host=False, goal=False),
        # many scenes solved together (training data, multi-query planning):
        # log-uniform sizes, mixed dimensions, ragged members
        dict(name="batch_24", kind="batch", members=24, n_min=1_000, n_max=50_000),
        # a control loop re-evaluating a policy with no allocation, odd size
        dict(name="evaluate_200k", kind="evaluate", n=200_003, window=0.1),
        # building the roadmap of one training scene on the GPU
        dict(name="roadmap_2d_100k", kind="roadmap", n=100_000, dim=2, k=63),
        # one chunk of a planner's mixed samples for one scene
        dict(name="sample_64k", kind="sample", rows=65_536, scenes=1),
        # bulk sampling over many scenes, a ragged last tile
        dict(name="forward_1m", kind="forward", rows=1_000_003, scenes=32),
        # one training step at the sizes training runs with
        dict(name="train_32x64x16", kind="train", scenes=32, targets=64, draws=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["schedule", "schedule", "schedule", "policy", "batch", "evaluate",
                       "roadmap", "sample", "forward", "train"])
    if kind == "schedule":
        dim = rng.choice([2, 3, 4, 6, 6, 7])
        n = _log(rng, 3_000, 150_000 if dim == 2 else 1_000_000)
        k = W.knn_k(n) if dim == 2 else rng.choice([20, 30, 37])
        blocks = _log(rng, 1, 40)
        return dict(kind=kind, n=n, dim=dim, k=k, block=-(-n // blocks),
                    f64=rng.random() < 0.25, host=rng.random() < 0.3, goal=rng.random() < 0.3)
    if kind == "policy":
        return dict(kind=kind, n=_log(rng, 300, 20_000), dim=rng.choice([2, 3]), k=30,
                    f64=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind=kind, members=rng.randint(3, 24), n_min=_log(rng, 300, 3_000),
                    n_max=_log(rng, 5_000, 50_000))
    if kind == "evaluate":
        return dict(kind=kind, n=_log(rng, 100, 262_144), window=rng.choice([0.03, 0.1, 0.5, 1.0]))
    if kind == "roadmap":
        dim = rng.choice([2, 2, 3, 6])
        n = _log(rng, 1_000, 100_000)
        return dict(kind=kind, n=n, dim=dim, k=W.knn_k(n) if dim == 2 else rng.choice([10, 30, 37]))
    if kind == "train":
        return dict(kind=kind, scenes=rng.randint(2, 32), targets=rng.randint(5, 64),
                    draws=rng.randint(2, 16))
    return dict(kind=kind, rows=_log(rng, 50, 1_000_000), scenes=rng.randint(1, 32))


# ---------------------------------------------------------------------------
# inputs

def _scene(rng, dim):
    """The unit square with 200 circles, or [-pi, pi]^dim with 64 balls; x_init
    (and in 2-D x_goal) kept free."""
    lo, hi, n_obs, r0, r1 = (0.0, 1.0, 200, 0.01, 0.04) if dim == 2 else (-PI, PI, 64, 0.3, 0.8)
    keep = [np.array([0.05, 0.05]), np.array([0.95, 0.95])] if dim == 2 else []
    c, r = np.empty((n_obs, dim)), np.empty(n_obs)
    for i in range(n_obs):
        while True:
            c[i], r[i] = rng.uniform(lo, hi, dim), rng.uniform(r0, r1)
            if all(np.sum((p - c[i]) ** 2) >= r[i] * r[i] for p in keep):
                break
    return W.Scene(dim, lo, hi, c, r)


def _points(rng, scene, n, seed):
    if scene.dim != 2:
        return GG.sample(scene, n, seed)[0]
    head = torch.tensor([[0.05, 0.05], [0.95, 0.95]], dtype=torch.float64, device="cuda")
    return torch.cat([head, GG.sample(scene, n - 2, seed)[0]])


def _roadmap(dim, n, k, seed, f64=False):
    rng = np.random.default_rng([int(seed), n, dim])
    scene = _scene(rng, dim)
    pts = _points(rng, scene, n, int(seed) * 1_000_003 + n)
    nbr = GG.knn(pts, scene.lo, scene.hi, min(k, n - 1))
    u, v, c, start = GG.edges(pts, nbr, scene, dim == 2, 16, np.float64 if f64 else np.float32)
    return pts, u, v, c, start


def _members(case, seed):
    rng = np.random.default_rng([case["members"], case["n_min"], case["n_max"]])
    sizes = np.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"]),
                               case["members"])).round().astype(int)
    dims = rng.choice([2, 3, 4, 6, 7], case["members"])
    return [_roadmap(int(d), int(n), W.knn_k(int(n)), int(seed) * 1000 + i)
            for i, (n, d) in enumerate(zip(sizes, dims))]


def _bfs_parents(n, u, v):
    """Breadth-first parents from vertex 0 (one level at a time on the device),
    each vertex taking the smallest neighbour of the level before."""
    src, dst = torch.cat([u, v]).long(), torch.cat([v, u]).long()
    depth = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    depth[0] = 0
    parent = torch.full((n,), n, dtype=torch.int64, device="cuda")
    for d in range(n):
        hit = (depth[src] == d) & (depth[dst] < 0)
        if not bool(hit.any()):
            break
        parent.scatter_reduce_(0, dst[hit], src[hit], "amin")
        depth[dst[hit]] = d + 1
    return torch.where(depth > 0, parent, torch.full_like(parent, -1)).int()


def _tree(case, seed):
    """A policy with ids in random order: each vertex's parent lies within the
    last `window` share of the vertices before it, one in 10^4 is unreached."""
    n = case["n"]
    gen = torch.Generator("cuda").manual_seed(int(seed))
    r = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
    i = torch.arange(n, device="cuda", dtype=torch.float64)
    par = torch.clamp((i * (1.0 - case["window"] * r)).long(), max=n - 1)
    par = torch.minimum(par, torch.clamp(torch.arange(n, device="cuda") - 1, min=0))
    perm = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"),
                      1 + torch.randperm(n - 1, generator=gen, device="cuda")])
    parent = torch.empty(n, dtype=torch.int32, device="cuda")
    parent[perm] = perm[par].int()
    parent[torch.rand(n, generator=gen, device="cuda") < 1e-4] = -1
    parent[0] = -1
    cost = 1e-3 + torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
    return parent, cost


def _weights(gen):
    """He-uniform parameters with small biases, in the packed order."""
    def uni(count, lim):
        return (2.0 * torch.rand(count, generator=gen, device="cuda") - 1.0) * lim
    l1, l2 = math.sqrt(6.0 / 4104), math.sqrt(6.0 / 256)
    return torch.cat([uni(256 * 4096, l1), uni(256 * 8, 0.4), uni(256, 0.05), uni(256 * 256, l2),
                      uni(256, 0.05), uni(2 * 256, l2), uni(2, 0.05)])


def _network_inputs(case, seed, rows):
    gen = torch.Generator("cuda").manual_seed(int(seed) * 7919 + rows)
    s = case["scenes"]
    x = dict(w=_weights(gen))
    x["grids"] = (torch.rand((s, 4096), generator=gen, device="cuda") < 0.3).float()
    x["noise"] = torch.randn((rows, 8), generator=gen, device="cuda")
    if case["kind"] == "train":
        t = s * case["targets"]
        x["scene"] = torch.arange(s, dtype=torch.int32, device="cuda").repeat_interleave(case["targets"])
        x["targets"] = torch.rand((t, 2), generator=gen, device="cuda")
        return x
    x["scene"] = torch.randint(0, s, (rows,), generator=gen, device="cuda", dtype=torch.int32)
    if case["kind"] == "sample":
        x["uniform"] = torch.rand((rows, 2), generator=gen, device="cuda")
        x["coin"] = torch.rand(rows, generator=gen, device="cuda")
    return x


def _rows(case):
    return case["scenes"] * case["targets"] * case["draws"] if case["kind"] == "train" else case["rows"]


# The rate at the far end of a decayed schedule.  A first Adam step moves every
# weight by about the rate whatever its gradient, so the rate sets how far a
# weight whose gradient is next to nothing may land.
LR = 3e-6


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("schedule", "policy"):
        n = case["n"]
        pts, u, v, c, start = _roadmap(case["dim"], n, case["k"], seed, case["f64"])
        st["g"] = torch.empty(n, dtype=torch.float64, device="cuda")
        st["p"] = torch.empty(n, dtype=torch.int32, device="cuda")
        st["graph"] = pkg.Graph(n, int(u.numel()), 0, np.float64 if case["f64"] else np.float32)
        if kind == "policy":
            st["edges"] = (u, v, c)
            st["init"] = _bfs_parents(n, u, v)
            return st
        if case["goal"]:
            goal = 1 if case["dim"] == 2 else int(
                torch.linalg.vector_norm(pts + pts[0], dim=1)[:max(2, n // 4)].argmin())
            h = 0.99 * torch.linalg.vector_norm(pts - pts[goal], dim=1)
            st["graph"].set_goal(goal, h.float().cpu().numpy())
        s, blocks = case["block"], []
        if case["host"]:
            u, v, c = u.cpu().pin_memory(), v.cpu().pin_memory(), c.cpu().pin_memory()
        for v0 in range(0, n, s):
            v1 = min(n, v0 + s)
            e0, e1 = int(start[v0]), int(start[v1])
            blocks.append((v1 - v0, u[e0:e1], v[e0:e1], c[e0:e1]))
        st["blocks"] = blocks
    elif kind == "batch":
        m = _members(case, seed)
        sizes = [int(x[0].shape[0]) for x in m]
        st["members"] = [x[1:4] for x in m]
        st["batch"] = pkg.Batch(sizes, [int(x[1].numel()) for x in m])
        st["at"] = np.r_[0, np.cumsum(sizes)]
        st["g"] = torch.empty(int(st["at"][-1]), dtype=torch.float64, device="cuda")
        st["p"] = torch.empty(int(st["at"][-1]), dtype=torch.int32, device="cuda")
    elif kind == "evaluate":
        st["parent"], st["cost"] = _tree(case, seed)
        st["g"] = torch.empty(case["n"], dtype=torch.float64, device="cuda")
    elif kind == "roadmap":
        rng = np.random.default_rng([int(seed), case["n"], case["dim"]])
        st["scene"] = _scene(rng, case["dim"])
        st["pts"] = _points(rng, st["scene"], case["n"], int(seed) * 1_000_003 + case["n"])
        # the program's own edge arrays, sized before the edge count is known
        cap = case["n"] * min(case["k"], case["n"] - 1)
        st["u"], st["v"] = torch.zeros((2, cap), dtype=torch.int32, device="cuda")
        st["cost"] = torch.zeros(cap, device="cuda")
    else:
        rows = _rows(case)
        st.update(_network_inputs(case, seed, rows))
        st["net"] = pkg.Proposal(case["scenes"], rows)
        st["net"].set_weights(st["w"])
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "schedule":
        g = st["graph"]
        g.reset()
        blocks, rounds = st["blocks"], []
        for b, (n_new, u, v, c) in enumerate(blocks):
            g.insert_batch(n_new, u, v, c)
            if case["host"] and b + 1 < len(blocks):
                g.prefetch_batch(*blocks[b + 1][1:])
            r = g.exploit()
            rounds.append((r["iterations"], r["switches"]))
        g.get_costs(st["g"])
        g.get_parents(st["p"])
        return dict(g=st["g"], p=st["p"], rounds=np.array(rounds, dtype=np.int64))
    if kind == "policy":
        g = st["graph"]
        g.reset()
        g.insert_batch(case["n"], *st["edges"])
        g.set_policy(st["init"])
        r = g.exploit()
        g.get_costs(st["g"])
        g.get_parents(st["p"])
        return dict(g=st["g"], p=st["p"],
                    rounds=np.array([r["iterations"], r["switches"]], dtype=np.int64))
    if kind == "batch":
        b, at = st["batch"], st["at"]
        b.reset()
        for i, (u, v, c) in enumerate(st["members"]):
            b.insert(i, u, v, c)
        r = b.exploit()
        for i in range(len(st["members"])):
            n = int(at[i + 1] - at[i])
            b.get_costs(i, n, st["g"][at[i]:at[i + 1]])
            b.get_parents(i, n, st["p"][at[i]:at[i + 1]])
        return dict(g=st["g"], p=st["p"],
                    rounds=np.array([r["iterations"], r["switches"]], dtype=np.int64))
    if kind == "evaluate":
        return dict(g=st["g"], status=pkg.pirrt_evaluate_noalloc(st["parent"], st["cost"], st["g"]))
    if kind == "roadmap":
        s = st["scene"]
        nbr = GG.knn(st["pts"], s.lo, s.hi, min(case["k"], case["n"] - 1))
        u, v, c, start = GG.edges(st["pts"], nbr, s, case["dim"] == 2, 16, np.float32)
        m = u.numel()
        st["u"][:m], st["v"][:m], st["cost"][:m] = u, v, c
        return dict(nbr=nbr, u=st["u"], v=st["v"], cost=st["cost"], start=start)
    net = st["net"]
    if kind == "train":
        loss = net.train_step(st["grids"], st["scene"], st["targets"], case["draws"], st["noise"], LR)
        return dict(loss=loss, weights=net.get_weights())
    if kind == "sample":
        return dict(xy=net.sample(st["grids"], st["scene"], st["noise"], st["uniform"], st["coin"], 0.5))
    return dict(xy=net.forward(st["grids"], st["scene"], st["noise"]))


# ---------------------------------------------------------------------------
# what no implementation can do without: every input read once, every output
# written once; each undirected edge formed once in each direction (an addition
# and a comparison); 2 operations per weight and row of the network.  Edge
# counts are about 0.57 k per vertex (the union of both directions' k nearest,
# less the edges an obstacle blocks).

PARAMS = 1_117_186
ROW_FLOPS = 2 * (8 * 256 + 256 * 256 + 256 * 2)


def _edges(n, k):
    return 0.57 * n * min(k, n - 1)


def work(case):
    kind = case["kind"]
    if kind in ("schedule", "policy"):
        m = _edges(case["n"], case["k"])
        return dict(bytes=m * (16 if case["f64"] else 12) + 12 * case["n"] + (4 * case["n"] if kind == "policy" else 0),
                    flops=4 * m)
    if kind == "batch":
        mean = (case["n_max"] - case["n_min"]) / math.log(case["n_max"] / case["n_min"])
        n = case["members"] * mean
        m = _edges(n, W.knn_k(int(mean)))
        return dict(bytes=12 * m + 12 * n, flops=4 * m)
    if kind == "evaluate":
        return dict(bytes=20 * case["n"], flops=case["n"])
    if kind == "roadmap":
        n, k, d = case["n"], min(case["k"], case["n"] - 1), case["dim"]
        m = _edges(n, k)
        return dict(bytes=8 * d * n + 4 * n * k + 12 * m + 8 * n, flops=3 * d * (n * k + m))
    rows, s = _rows(case), case["scenes"]
    fwd = rows * ROW_FLOPS + s * 2 * 4096 * 256
    if kind == "train":
        t = s * case["targets"]
        return dict(bytes=rows * 32 + t * 12 + s * 4096 * 4 + 7 * 4 * PARAMS,
                    flops=fwd + t * 2 * ROW_FLOPS + s * 2 * 4096 * 256)
    return dict(bytes=rows * (32 + 4 + 8 + (12 if kind == "sample" else 0)) + s * 4096 * 4 + 4 * PARAMS,
                flops=fwd)


# ---------------------------------------------------------------------------
# the same results in 64 bits

def _distances(n, u, v, c, roots):
    """Shortest-path costs from the roots: Bellman-Ford sweeps."""
    src, dst = torch.cat([u, v]).long(), torch.cat([v, u]).long()
    w = torch.cat([c, c]).double()
    g = torch.full((n,), math.inf, dtype=torch.float64, device="cuda")
    g[roots] = 0.0
    while True:
        old = g.clone()
        g.scatter_reduce_(0, dst, old[src] + w, "amin")
        if torch.equal(g, old):
            return g


def _mlp64(w, grids, scene, z):
    o = np.cumsum([0, 256 * 4096, 256 * 8, 256, 256 * 256, 256, 2 * 256, 2])
    p = [w[o[i]:o[i + 1]] for i in range(7)]
    a1 = (grids @ p[0].view(256, 4096).T)[scene] + z @ p[1].view(256, 8).T + p[2]
    a2 = torch.relu(a1) @ p[3].view(256, 256).T + p[4]
    return torch.sigmoid(torch.relu(a2) @ p[5].view(2, 256).T + p[6])


def _forward64(x, rows):
    out = [_mlp64(x["w"].double(), x["grids"].double(), x["scene"][i:i + 131072].long(),
                  x["noise"][i:i + 131072].double()) for i in range(0, rows, 131072)]
    return torch.cat(out)


def _train64(case, x):
    t, k = x["targets"].shape[0], case["draws"]
    w = x["w"].double()
    grids, tg, z = x["grids"].double(), x["targets"].double(), x["noise"].double()
    scene = x["scene"].long()
    with torch.no_grad():
        y = _mlp64(w, grids, scene.repeat_interleave(k), z).view(t, k, 2)
        pick = ((y - tg[:, None]) ** 2).sum(2).argmin(1)
    w = w.clone().requires_grad_(True)
    y = _mlp64(w, grids, scene, z.view(t, k, 8)[torch.arange(t, device="cuda"), pick])
    loss = ((y - tg) ** 2).sum(1).mean()
    (gr,) = torch.autograd.grad(loss, w)
    return float(loss), (w - LR * gr / (gr.abs() + 1e-8)).detach()


def _edge_costs64(case, st):
    """FP64 lengths of the roadmap's edges in its order (larger endpoint, then
    smaller): brute-force neighbours by FP32 squared distance, then id; edges of
    either direction; those that meet no obstacle."""
    s, pts, n, dim = st["scene"], st["pts"], case["n"], case["dim"]
    k, q = min(case["k"], case["n"] - 1), st["pts"].float()
    nbr, step = [], max(1, 200_000_000 // n)
    for i in range(0, n, step):
        d2 = torch.zeros((min(step, n - i), n), device="cuda")
        for d in range(dim):
            t = q[i:i + step, d, None] - q[None, :, d]
            d2 += t * t
        key = (d2.view(torch.int32).long() << 32) + torch.arange(n, device="cuda")
        key[torch.arange(len(key), device="cuda"), torch.arange(i, i + len(key), device="cuda")] = 1 << 62
        nbr.append(torch.topk(key, k, dim=1, largest=False).values & 0xFFFFFFFF)
    j = torch.cat(nbr).reshape(-1)
    i = torch.arange(n, device="cuda").repeat_interleave(k)
    e = torch.unique(torch.maximum(i, j) * n + torch.minimum(i, j))
    a, b = pts[e % n], pts[e // n]
    ok = torch.ones(len(e), dtype=torch.bool, device="cuda")
    for c, r in zip(torch.from_numpy(s.centers).cuda(), s.radii):
        if dim == 2:
            ab = b - a
            t = (((c - a) * ab).sum(1) / (ab * ab).sum(1)).clamp(0.0, 1.0)
            ok &= ((a + t[:, None] * ab - c) ** 2).sum(1) >= r * r
        else:
            for f in range(16):
                ok &= ((a + f / 15 * (b - a) - c) ** 2).sum(1) >= r * r
    return ((b - a)[ok] ** 2).sum(1).sqrt()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("schedule", "policy"):
        if kind == "schedule" and case["goal"]:
            return None  # costs below pruned vertices may stay above their path's
        n = case["n"]
        _, u, v, c, _ = _roadmap(case["dim"], n, case["k"], seed, case["f64"])
        return dict(g=_distances(n, u, v, c, [0]), p=None, rounds=None)
    if kind == "batch":
        at, parts, roots = 0, [], []
        for pts, u, v, c, _ in _members(case, seed):
            parts.append((u.long() + at, v.long() + at, c))
            roots.append(at)
            at += int(pts.shape[0])
        u, v, c = (torch.cat(x) for x in zip(*parts))
        return dict(g=_distances(at, u, v, c, roots), p=None, rounds=None)
    if kind == "evaluate":
        parent, cost = _tree(case, seed)
        g = torch.full((case["n"],), math.inf, dtype=torch.float64, device="cuda")
        g[0] = 0.0
        live = (parent >= 0).nonzero().squeeze(1)
        while len(live):
            val = g[parent[live].long()] + cost[live]
            done = torch.isfinite(val)
            if not bool(done.any()):
                break
            g[live[done]] = val[done]
            live = live[~done]
        return dict(g=g, status=None)
    if kind == "roadmap":
        st = prepare(case, seed)
        c = _edge_costs64(case, st)
        cost = torch.cat([c, c.new_zeros(st["cost"].numel() - len(c))])
        return dict(nbr=None, u=None, v=None, cost=cost, start=None)
    rows = _rows(case)
    x = _network_inputs(case, seed, rows)
    if kind == "train":
        loss, w = _train64(case, x)
        return dict(loss=loss, weights=w)
    y = _forward64(x, rows)
    if kind == "sample":
        y = torch.where((x["coin"] < 0.5)[:, None], y, x["uniform"].double())
    return dict(xy=y)
