"""Timed cases: the work a user has the library do, through its public calls.

Every case runs on the graph families of the benchmark and the tests: sparse
Erdos-Renyi graphs ("er"), road-shaped perturbed grids ("grid": a W x H grid, a
random spanning tree kept, a quarter of the edges deleted) and Chung-Lu
power-law graphs ("cl", exponent 2.1).  ``work`` counts a departure of
Wilson's walk as 70 integer operations (a ten-round Philox block, the bounded
draw and the word update) and a vertex of a finished tree as 20 (sizes,
volumes, preorder and its share of f).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2511_16356_gb300 import kc
from paper_2511_16356_gb300 import synth

OPS_PER_DEPARTURE = 70
OPS_PER_VERTEX = 20


def listed():
    return [
        # The smallest call in use: a small graph, a few dozen trees (latency and launches).
        {"name": "er300 sample 64", "kind": "sample", "family": "er", "n": 300, "deg": 6.0,
         "trees": 64},
        # The small static configuration: 2000 trees on a sparse random graph of 2000 vertices.
        {"name": "er2000 sample 2000", "kind": "sample", "family": "er", "n": 2000, "deg": 8.0,
         "trees": 2000},
        # Time to a relative error: pilot, stopping rule and the batches it asks for.
        {"name": "er2000 estimate 1%", "kind": "estimate", "family": "er", "n": 2000, "deg": 8.0,
         "eps": 0.01, "delta": 0.05},
        # Road-shaped graph under the default options (the profiled grid).
        {"name": "grid300 sample 1000", "kind": "sample", "family": "grid", "n": 90000, "deg": 3.0,
         "trees": 1000},
        # Road-shaped graph with rejection by walk length, thousands of trees in one wave: the
        # options of the headline run.
        {"name": "grid350 reject 3000", "kind": "reject", "family": "grid", "n": 122500,
         "deg": 3.0, "trees": 3000, "cap_per_vertex": 13.0, "accept": 0.65},
        # Large power-law graph: the social-network configuration.
        {"name": "cl2m sample 384", "kind": "sample", "family": "cl", "n": 2000000, "deg": 17.0,
         "trees": 384},
        # A user with a new graph: handle from host arrays, a short estimate's trees, results read.
        {"name": "cl300k create 128", "kind": "create", "family": "cl", "n": 300000, "deg": 17.0,
         "trees": 128},
        # Dynamic graph, ISM: a batch of insertions and deletions on a retained pool.
        {"name": "cl100k ism 1000", "kind": "update", "family": "cl", "n": 100000, "deg": 20.0,
         "trees": 1000, "mode": "ism", "edges": 2},
        # The same maintenance by BSM (resampling).
        {"name": "cl30k bsm 500", "kind": "update", "family": "cl", "n": 30000, "deg": 20.0,
         "trees": 500, "mode": "bsm", "edges": 2},
        # Many graphs of uneven size in one call (the batched configuration).
        {"name": "multi 24 graphs", "kind": "multi", "graphs": 24, "nmax": 20000, "trees": 256},
        # Concurrent queries on resident graphs through the server.
        {"name": "serve 24 queries", "kind": "serve", "graphs": 12, "nmax": 20000, "queries": 24,
         "eps": 0.03, "delta": 0.05},
        # Sampling without allocation into the caller's tensors.
        {"name": "er2000 noalloc 2000", "kind": "noalloc", "family": "er", "n": 2000, "deg": 8.0,
         "trees": 2000},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["sample", "sample", "sample", "reject", "estimate", "create", "update",
                       "multi", "serve", "noalloc"])
    family = rng.choice(["er", "grid", "cl"])
    if kind in ("sample", "create"):
        # up to the work of the largest listed case of the family
        top = {"er": 1000000, "grid": 90000, "cl": 2000000}[family]
        n = log_int(300, top if kind == "sample" else top // 6)
        most = {"er": 4.0e8, "grid": 9.0e7, "cl": 7.0e8}[family] / n
        trees = log_int(33, max(64, min(4000, most)))
        if kind == "create":
            trees = max(33, trees // 8)
        deg = {"er": rng.uniform(6, 12), "grid": 3.0, "cl": rng.uniform(10, 20)}[family]
        return {"kind": kind, "family": family, "n": n, "deg": deg, "trees": trees}
    if kind == "reject":
        n = log_int(2500, 122500)
        return {"kind": kind, "family": "grid", "n": n, "deg": 3.0,
                "trees": log_int(200, max(400, min(6000, 3.6e8 / n))),
                "cap_per_vertex": 0.4 + 1.05 * math.log(n), "accept": 0.65}
    if kind == "estimate":
        n = log_int(300, 20000)
        return {"kind": kind, "family": "er", "n": n, "deg": rng.uniform(6, 12),
                "eps": rng.choice([0.05, 0.02, 0.01]), "delta": rng.choice([0.05, 0.01])}
    if kind == "update":
        mode = rng.choice(["ism", "bsm"])
        n = log_int(2000, 100000 if mode == "ism" else 30000)
        return {"kind": kind, "family": rng.choice(["er", "cl"]), "n": n,
                "deg": rng.uniform(10, 20), "trees": log_int(64, 1000), "mode": mode,
                "edges": rng.randint(1, 2)}
    if kind == "multi":
        return {"kind": kind, "graphs": rng.randint(2, 24), "nmax": log_int(2000, 20000),
                "trees": log_int(32, 256)}
    if kind == "serve":
        return {"kind": kind, "graphs": rng.randint(3, 12), "nmax": log_int(2000, 20000),
                "queries": rng.randint(6, 24), "eps": rng.choice([0.05, 0.03]), "delta": 0.05}
    n = log_int(300, 4000)
    return {"kind": "noalloc", "family": "er", "n": n, "deg": rng.uniform(6, 12),
            "trees": log_int(64, min(2000, (8 << 20) // n))}


# ---------------------------------------------------------------- inputs

def _random_graph(n, mean_deg, seed, gamma=0.0):
    """n vertices, endpoints drawn on the GPU: uniformly, or with gamma with probability
    proportional to (i + i0)^(-1/(gamma-1)) scaled to the mean degree with largest weight
    sqrt(n mean_deg); repeats and loops dropped, every other component joined to the largest
    by one edge."""
    dev = "cuda"
    i = torch.arange(n, dtype=torch.float64, device=dev)
    a = 1.0 / (gamma - 1.0) if gamma else 0.0
    lo, hi = 1e-6, float(n)
    for _ in range(60 if gamma else 0):
        mid = math.sqrt(lo * hi)
        x = (i + mid) ** (-a)
        if float(x[0] / x.mean()) > math.sqrt(n / mean_deg):
            lo = mid
        else:
            hi = mid
    cum = torch.cumsum((i + hi) ** (-a), 0)
    gen = torch.Generator(device=dev).manual_seed(seed)
    ends = torch.rand(2, int(n * mean_deg / 2), dtype=torch.float64, device=dev, generator=gen)
    u, v = torch.searchsorted(cum, ends * cum[-1]).clamp_(max=n - 1)
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.cat([u * n + v, v * n + u]))
    label = torch.arange(n, device=dev)
    while True:
        new = label.scatter_reduce(0, key // n, label[key % n], "amin")
        new = new[new]
        if torch.equal(new, label):
            break
        label = new
    inside = label == torch.bincount(label).argmax()
    rest, core = torch.unique(label[~inside]), inside.nonzero()[:, 0]
    to = core[torch.randint(core.numel(), rest.shape, device=dev, generator=gen)]
    key = torch.unique(torch.cat([key, rest * n + to, to * n + rest]))
    row = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    row[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    return synth.Graph(row.cpu().numpy(), (key % n).to(torch.int32).cpu().numpy(), "random%d" % n)


def _graph(family, n, deg, seed):
    if family == "er":
        return synth.er_lcc(n, min(1.0, deg / (n - 1)), seed)
    if family == "grid":
        w = max(8, int(math.sqrt(n)))
        return synth.grid_perturbed(w, max(8, n // w), 0.25, seed)
    return _random_graph(n, deg, seed, 2.1)


def _mixed(count, nmax, seed):
    """The serving mix: the three families in turn, sizes log-uniform on [1000, nmax]."""
    rng = np.random.default_rng(seed)
    sizes = np.exp(rng.uniform(math.log(1000.0), math.log(float(nmax)), count)).astype(int)
    fam = ("er", "grid", "cl")
    return [_graph(fam[k % 3], int(sizes[k]), (8.0, 3.0, 10.0)[k % 3], seed + 1 + k)
            for k in range(count)]


def _config(**kw):
    cfg = kc.kc_config_default()
    cfg.keep_trees = 0
    for k, v in kw.items():
        setattr(cfg, k, v)
    return cfg


def _ops(g, p0, count, seed):
    """Insertions of absent pairs and deletions of edges on a triangle that are not path-tree
    edges, every change undone by the end of the batch."""
    rng = np.random.default_rng(seed)
    rows = [None] * g.n

    def nbrs(u):
        if rows[u] is None:
            rows[u] = set(int(x) for x in g.neighbors(u))
        return rows[u]

    new, old = [], []
    while len(new) < count:
        u, v = (int(x) for x in rng.integers(0, g.n, 2))
        if u != v and v not in nbrs(u) and (u, v) not in new and (v, u) not in new:
            new.append((u, v))
    tries = 0
    while len(old) < count:
        u = int(rng.integers(0, g.n))
        v = int(rng.choice(sorted(nbrs(u))))
        tries += 1
        plain = p0[u] != v and p0[v] != u and (u, v) not in old and (v, u) not in old
        # a sparse graph may have few triangles: then any edge between vertices of degree >= 3
        if plain and (nbrs(u) & nbrs(v) or (tries > 200 and min(len(nbrs(u)), len(nbrs(v))) > 2)):
            old.append((u, v))
    ops = []
    for a, b in zip(new, old):
        ops += [(a[0], a[1], kc.KC_OP_INSERT), (b[0], b[1], kc.KC_OP_DELETE)]
    for a, b in zip(new, old):
        ops += [(b[0], b[1], kc.KC_OP_INSERT), (a[0], a[1], kc.KC_OP_DELETE)]
    return ops


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "seed": 1000 + seed}
    if kind in ("multi", "serve"):
        graphs = _mixed(case["graphs"], case["nmax"], 17 * seed + 5)
        if kind == "multi":
            s["graphs"] = [kc.KemenyGraph.from_graph(g, _config()) for g in graphs]
        else:
            s["server"] = kc.Server(workers=4, coalesce=1)
            s["ids"] = [s["server"].add_graph(g, _config()) for g in graphs]
        return s
    if kind in ("update", "noalloc") and case["family"] == "er":
        # results have one entry per vertex: every seed's graph has exactly n of them
        g = _random_graph(case["n"], case["deg"], 17 * seed + 5)
    else:
        g = _graph(case["family"], case["n"], case["deg"], 17 * seed + 5)
    if kind == "create":
        s["host"] = g
    elif kind == "reject":
        s["graph"] = kc.KemenyGraph.from_graph(
            g, _config(reject_steps=int(case["cap_per_vertex"] * g.n),
                       reject_accept_hint=case["accept"]))
    elif kind == "update":
        G = s["graph"] = kc.KemenyGraph.from_graph(g, _config(keep_trees=1))
        G.sample(s["seed"], case["trees"])
        s["ops"] = _ops(g, G.tau0()["p0"], case["edges"], seed)
        s["mode"] = kc.KC_UPDATE_ISM if case["mode"] == "ism" else kc.KC_UPDATE_BSM
    elif kind == "noalloc":
        with kc.KemenyGraph.from_graph(g, _config()) as G:
            s["root"] = G.tau0()["root"]
        s["row_off"], s["col"] = torch.from_numpy(g.row_off).cuda(), torch.from_numpy(g.col).cuda()
        s["parent"] = torch.empty(case["trees"], g.n, dtype=torch.int32, device="cuda")
        s["steps"] = torch.empty(case["trees"], dtype=torch.int64, device="cuda")
        s["status"] = torch.empty(1, dtype=torch.int32, device="cuda")
    else:
        s["graph"] = kc.KemenyGraph.from_graph(g, _config())
    return s


# ---------------------------------------------------------------- one pass

def _results(G, estimate):
    got = G.samples()
    return {"f": got["f"], "steps": got["steps"], "sid": got["sid"], "K": estimate}


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind in ("sample", "reject"):
        G = s["graph"]
        G.reset(s["seed"])
        G.sample(s["seed"], case["trees"])
        return _results(G, G.estimate())
    if kind == "estimate":
        G = s["graph"]
        G.reset(s["seed"])
        # the stopping rule decides how many trees: the estimate and the moments behind it
        estimate = G.estimate(case["eps"], case["delta"])
        sums = G.pool_sums()
        return {"K": estimate, "trees": sums["count"], "wf": sums["wf_sum"], "x2": sums["x2_sum"]}
    if kind == "create":
        with kc.KemenyGraph.from_graph(s["host"], _config()) as G:
            G.sample(s["seed"], case["trees"])
            return _results(G, G.estimate())
    if kind == "update":
        G = s["graph"]
        G.update(s["ops"], s["mode"])
        got = G.samples()
        tree = G.tree(case["trees"] // 2)
        return {"f": got["f"], "w": got["w"], "steps": got["steps"], "sid": got["sid"],
                "K": G.estimate(), "tree": {k: tree[k] for k in ("parent", "depth", "din", "vol")}}
    if kind == "multi":
        for G in s["graphs"]:
            G.reset(s["seed"])
        kc.kc_sample_multi([G.h for G in s["graphs"]], [s["seed"]] * len(s["graphs"]),
                           [case["trees"]] * len(s["graphs"]))
        got = [G.samples() for G in s["graphs"]]
        return {"f": np.concatenate([x["f"] for x in got]),
                "steps": np.concatenate([x["steps"] for x in got])}
    if kind == "serve":
        ids, srv = s["ids"], s["server"]
        tickets = [srv.query(ids[q % len(ids)], s["seed"] + q, case["eps"], case["delta"])
                   for q in range(case["queries"])]
        infos = [srv.wait(t) for t in tickets]
        return {"K": np.array([x["K"] for x in infos]),
                "trees": np.array([x["trees"] for x in infos], dtype=np.int64)}
    lib = kc.load()
    st = lib.kc_wilson_noalloc(s["row_off"].shape[0] - 1, s["row_off"].data_ptr(),
                               s["col"].data_ptr(), s["root"], s["seed"], 0, case["trees"], 0,
                               s["parent"].data_ptr(), s["steps"].data_ptr(),
                               s["status"].data_ptr(), torch.cuda.current_stream().cuda_stream)
    if st != kc.KC_OK:
        raise RuntimeError(kc.kc_status_string(st))
    return {"parent": s["parent"], "steps": s["steps"], "status": s["status"]}


# ---------------------------------------------------------------- what a pass needs

def _departures(family, n):
    """Mean departures of one tree, from runs of the oracle."""
    return n * {"er": 1.6, "grid": 1.1 * math.log(n), "cl": 1.1}[family]


def work(case):
    kind = case["kind"]
    if kind in ("multi", "serve"):
        n = (case["nmax"] - 1000) / math.log(case["nmax"] / 1000.0)  # mean of the log-uniform size
        trees = case["graphs"] * case["trees"] if kind == "multi" else case["queries"] * 128
        per = sum(_departures(f, n) for f in ("er", "grid", "cl")) / 3
        return {"bytes": case["graphs"] * n * 56 + trees * 16,
                "flops": trees * (OPS_PER_DEPARTURE * per + OPS_PER_VERTEX * n)}
    n = case["n"]
    graph = 8 * (n + 1) + 4 * n * case["deg"]
    if kind == "noalloc":
        return {"bytes": graph + case["trees"] * (4 * n + 8),
                "flops": case["trees"] * OPS_PER_DEPARTURE * _departures(case["family"], n)}
    if kind == "update":
        # about one tree in six changes with an operation: its parents are read and written
        changed = 4 * case["edges"] * case["trees"] / 6
        per = OPS_PER_VERTEX * n
        if case["mode"] == "bsm":
            per += OPS_PER_DEPARTURE * _departures(case["family"], n)
        return {"bytes": graph + changed * 8 * n + case["trees"] * 32, "flops": changed * per}
    trees = case["trees"] if "trees" in case else 1024
    walked = trees / case["accept"] if kind == "reject" else trees
    return {"bytes": graph + trees * 32,
            "flops": walked * OPS_PER_DEPARTURE * _departures(case["family"], n) +
                     trees * OPS_PER_VERTEX * n}


# ---------------------------------------------------------------- K by plain torch, 64 bits

def _levels(n, src, dst, start):
    level = np.full(n, -1, dtype=np.int64)
    level[start] = 0
    lev = 0
    while True:
        nxt = dst[(level[src] == lev) & (level[dst] < 0)]
        if not nxt.size:
            return level
        lev += 1
        level[nxt] = lev


def _root(n, src, dst, deg):
    """Highest degree, ties broken towards the centre, smallest id among equals."""
    ties = np.flatnonzero(deg == deg.max())
    if ties.size == 1:
        return int(ties[0])
    a = int(_levels(n, src, dst, int(ties[0])).argmax())
    la = _levels(n, src, dst, a)
    b = int(la.argmax())
    lb = _levels(n, src, dst, b)
    lc = _levels(n, src, dst, int(np.minimum(la, lb).argmax()))
    far = np.maximum(np.maximum(la, lb), lc)[ties]
    return int(ties[far.argmin()])


def _philox(c0, c1, c2, seed):
    """Philox4x32-10 (Salmon et al.) on 32-bit values held in int64."""
    mask = 0xFFFFFFFF

    def mul(a, m):
        hi = ((a >> 16) * m + (((a & 0xFFFF) * m) >> 16)) >> 16
        return hi, (a * m) & mask

    c3 = torch.zeros_like(c0)
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        h0, l0 = mul(c0, 0xD2511F53)
        h1, l1 = mul(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c0, c1, c2, c3


def _arrow(v, count, sample, seed, row, deg, col):
    """The neighbour that v's departure number `count` takes (multiply and reject)."""
    s = deg[v]
    thr = (2 ** 32 - s) % s
    pick = torch.full_like(v, -1)
    for w in _philox(v, count, sample, seed):
        m = w * s
        pick = torch.where((pick < 0) & ((m & 0xFFFFFFFF) >= thr), m >> 32, pick)
    return col[row[v] + pick]


def _trees(row, deg, col, root, seed, count):
    """Parents [count, n]: every vertex shows its current arrow, the arrows of all cycles are
    replaced, until none is left."""
    n = deg.shape[0]
    v = torch.arange(n, device="cuda").repeat(count, 1)
    tree = torch.arange(count, device="cuda")
    used = torch.zeros_like(v)
    nxt = _arrow(v, used, tree[:, None].expand(-1, n), seed, row, deg, col)
    nxt[:, root] = root
    live = tree
    while live.numel():
        hop = nxt[live]
        for _ in range(max(1, math.ceil(math.log2(n)))):
            hop = hop.gather(1, hop)
        on = torch.zeros(hop.shape, dtype=torch.bool, device="cuda").scatter_(1, hop, True)
        on[:, root] = False
        r, x = on.nonzero(as_tuple=True)
        t = live[r]
        used[t, x] += 1
        nxt[t, x] = _arrow(x, used[t, x], t, seed, row, deg, col)
        live = live[on.any(1)]
    nxt[:, root] = -1
    return nxt


def _f_sum(par, deg, p0, root, twom):
    """Sum over the trees of f = sum_v d(v) Q(v), Q by the path-tree walk of every vertex."""
    B, n = par.shape
    up = par.clamp(min=0)
    depth = torch.zeros_like(par)
    x = par.clone()
    while bool((x >= 0).any()):
        depth += x >= 0
        x = torch.where(x >= 0, par.gather(1, x.clamp(min=0)), x)
    size = torch.ones_like(par)
    vol = deg.repeat(B, 1)
    top = int(depth.max())
    for d in range(top, 0, -1):
        r, c = (depth == d).nonzero(as_tuple=True)
        at = r * n + up[r, c]
        size.view(-1).index_add_(0, at, size[r, c])
        vol.view(-1).index_add_(0, at, vol[r, c])
    order = par.sort(dim=1, stable=True).indices
    run = size.gather(1, order).cumsum(1) - size.gather(1, order)
    p = par.gather(1, order)
    first = torch.ones_like(p, dtype=torch.bool)
    first[:, 1:] = p[:, 1:] != p[:, :-1]
    base = torch.where(first, run, torch.zeros_like(run)).cummax(1).values
    off = torch.empty_like(run).scatter_(1, order, run - base)
    din = torch.zeros_like(par)
    for d in range(1, top + 1):
        r, c = (depth == d).nonzero(as_tuple=True)
        din[r, c] = din[r, up[r, c]] + 1 + off[r, c]
    q = torch.zeros_like(par)
    x = torch.arange(n, device="cuda")
    while bool((x != root).any()):
        w = p0[x].clamp(min=0)  # the path-tree parent of x
        live = (x != root)[None, :]
        same = live & (par[:, x] == w)
        q += torch.where(same & (din[:, x] <= din) & (din < din[:, x] + size[:, x]),
                         twom - vol[:, x], 0)
        turned = live & ~same & (w != root)[None, :] & (par[:, w] == x)
        q -= torch.where(turned & (din[:, w] <= din) & (din < din[:, w] + size[:, w]),
                         twom - vol[:, w], 0)
        x = torch.where(x != root, w, x)
    q[:, root] = 0
    return int((q * deg).sum())


def exact(case, seed):
    """K of the small sampling cases; the other cases' trees take too long in plain torch."""
    if case["kind"] != "sample" or case["family"] != "er" or case["n"] * case["trees"] > 5000000:
        return None
    g = _graph(case["family"], case["n"], case["deg"], 17 * seed + 5)
    n, src, dst = g.n, np.repeat(np.arange(g.n), g.deg), g.col.astype(np.int64)
    root = _root(n, src, dst, g.deg)
    level = _levels(n, src, dst, root)
    p0 = np.full(n, n, dtype=np.int64)
    closer = level[dst] == level[src] - 1
    np.minimum.at(p0, src[closer], dst[closer])
    p0[root] = -1
    row, deg, col, p0 = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.int64)).cuda()
                         for a in (g.row_off[:-1], g.deg, dst, p0))
    total = 0
    par = _trees(row, deg, col, root, 1000 + seed, case["trees"])
    for part in par.split(500):
        total += _f_sum(part, deg, p0, root, 2 * g.m)
    return {"f": None, "steps": None, "sid": None, "K": total / (2 * g.m * case["trees"])}
