"""The calls that the library's speed is judged by, as a user's program makes them.

A case is one call (or one short sequence of calls) through the public entry points on one graph of
a size that the library meets: the paper's three graph classes (uniform random, R-MAT, road-like
grid), its three algorithms, the paper's modes and the automatic choice, several sources at once, a
batch over many graphs, and the load of a new graph.  ``listed`` names twelve of them, ``draw`` gives
others of the same ranges, ``prepare`` makes what the program holds before the call, ``run`` is the
call, ``work`` the bytes and operations that it cannot do without, and ``exact`` the result by plain
int64 relaxation in torch.
"""
from __future__ import annotations

import math

import torch

import paper_1903_01665_gb300 as fg

MODE = {"vertex_sync": fg.FG_VERTEX_SYNC, "vertex_async": fg.FG_VERTEX_ASYNC, "edge_sync": fg.FG_EDGE_SYNC,
        "edge_async": fg.FG_EDGE_ASYNC, "auto": fg.FG_AUTO}
ALGO = {"sssp": fg.FG_ALGO_SSSP, "bfs": fg.FG_ALGO_BFS, "cc": fg.FG_ALGO_CC}
INF = fg.FG_INF


def listed():
    big = {"family": "rmat", "n": 1 << 22}
    return [
        # one latency-bound query on a graph that fits in L2: a service that answers small questions
        {"name": "er16k_sssp_vertex_sync", "kind": "query", "family": "er", "n": 16384, "m": 131072,
         "algo": "sssp", "mode": "vertex_sync"},
        # the main workload: R-MAT 22.  SSSP in the default mode, in the edge-based one, and as picked
        {"name": "rmat22_sssp_vertex_sync", "kind": "query", **big, "algo": "sssp", "mode": "vertex_sync"},
        {"name": "rmat22_sssp_edge_sync", "kind": "query", **big, "algo": "sssp", "mode": "edge_sync"},
        {"name": "rmat22_sssp_auto", "kind": "query", **big, "algo": "sssp", "mode": "auto"},
        # reachability and components of the same social-network-like graph
        {"name": "rmat22_bfs_auto", "kind": "query", **big, "algo": "bfs", "mode": "auto"},
        {"name": "rmat22_cc_auto", "kind": "query", **big, "algo": "cc", "mode": "auto"},
        # routing on a road-like graph: hundreds of rounds, little work in each
        {"name": "grid4096_sssp_auto", "kind": "query", "family": "grid", "side": 4096, "whi": 10000,
         "algo": "sssp", "mode": "auto"},
        # hop counts on a smaller road-like graph of an odd side
        {"name": "grid1023_bfs_auto", "kind": "query", "family": "grid", "side": 1023, "whi": 10000,
         "algo": "bfs", "mode": "auto"},
        # a group of same-graph requests as a server fuses them: the smallest graph of the serving set,
        # whose state exceeds L2
        {"name": "rmat24_multi8_sssp", "kind": "multi", "family": "rmat", "n": 1 << 24, "algo": "sssp", "k": 8},
        # a smaller group on a graph of odd size
        {"name": "rmat3m_multi5_bfs", "kind": "multi", "family": "rmat", "n": 3000001, "algo": "bfs", "k": 5},
        # many queries over resident graphs of uneven size in one batch
        {"name": "batch_mixed12", "kind": "batch", "graphs": 12, "lo": 10, "hi": 20, "per_graph": 8},
        # a new edge list arrives on the device, is loaded, asked for its components and dropped
        {"name": "rmat22_load_cc", "kind": "load", **big, "form": "coo"},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "query", "query", "multi", "multi", "batch", "load"])
    if kind == "batch":
        lo = rng.randint(10, 13)
        return {"kind": "batch", "graphs": rng.randint(4, 12), "lo": lo, "hi": rng.randint(lo + 3, 20),
                "per_graph": rng.randint(3, 8)}
    family = rng.choice(["er", "rmat", "rmat", "grid"]) if kind != "load" else "rmat"
    case = {"kind": kind, "family": family}
    if family == "er":
        case["n"] = _logint(rng, 1000, 2000000)
        case["m"] = int(case["n"] * rng.uniform(4.0, 16.0))
    elif family == "rmat":
        case["n"] = _logint(rng, 1000, (1 << 24) if kind == "multi" else (1 << 22))
    else:
        case["side"] = _logint(rng, 33, 4096)
        case["whi"] = rng.choice([1000, 10000])
    if kind == "load":
        case["form"] = rng.choice(["coo", "csr"])
        return case
    if kind == "multi":
        case["algo"] = rng.choice(["sssp", "bfs"])
        case["k"] = rng.randint(2, 8)
        return case
    # components of a grid or a uniform graph are one giant one whatever the seed: asked of R-MAT only
    case["algo"] = rng.choice(["sssp", "sssp", "bfs", "cc"] if family == "rmat" else ["sssp", "sssp", "bfs"])
    case["mode"] = rng.choice(["vertex_sync", "vertex_async", "edge_sync", "edge_async", "auto", "auto"])
    return case


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _randint(gen, lo, hi, count):
    return torch.randint(lo, hi, (count,), generator=gen, device="cuda", dtype=torch.int32)


def _rmat(n, seed):
    """R-MAT .57/.19/.19/.05, 16 edges a vertex, weights U[1,1000]; ids scaled to n if it is no power of two."""
    gen = _gen(seed)
    bits = max(1, (n - 1).bit_length())
    m = 16 * n
    src = torch.empty(m, dtype=torch.int32, device="cuda")
    dst = torch.empty(m, dtype=torch.int32, device="cuda")
    step = 1 << 25
    for lo in range(0, m, step):
        cnt = min(step, m - lo)
        u = torch.zeros(cnt, dtype=torch.int32, device="cuda")
        v = torch.zeros(cnt, dtype=torch.int32, device="cuda")
        for _ in range(bits):
            r = torch.rand(cnt, generator=gen, device="cuda")
            u.mul_(2).add_(r >= 0.76)
            v.mul_(2).add_(((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
        if n & (n - 1):
            u = ((u.long() * n) >> bits).int()
            v = ((v.long() * n) >> bits).int()
        src[lo:lo + cnt] = u
        dst[lo:lo + cnt] = v
    return n, src, dst, _randint(gen, 1, 1001, m)


def _er(n, m, seed):
    """Uniform random directed edges without self-loops, weights U[1,100]."""
    gen = _gen(seed)
    src = _randint(gen, 0, n, m)
    dst = (src + _randint(gen, 1, n, m)) % n
    return n, src, dst, _randint(gen, 1, 101, m)


def _grid(side, whi, seed):
    """4-neighbour grid, 2 % of the pairs deleted, 0.1 % random shortcut pairs, both directions, weights U[1,whi]."""
    gen = _gen(seed)
    n = side * side
    ids = torch.arange(n, dtype=torch.int32, device="cuda").view(side, side)
    lo = torch.cat([ids[:, :-1].reshape(-1), ids[:-1].reshape(-1)])
    hi = torch.cat([ids[:, 1:].reshape(-1), ids[1:].reshape(-1)])
    keep = torch.rand(lo.numel(), generator=gen, device="cuda") >= 0.02
    short = int(round(0.001 * lo.numel()))
    su = _randint(gen, 0, n, short)
    sv = (su + _randint(gen, 1, n, short)) % n
    lo = torch.cat([lo[keep], su])
    hi = torch.cat([hi[keep], sv])
    src = torch.stack([lo, hi], 1).reshape(-1)
    dst = torch.stack([hi, lo], 1).reshape(-1)
    return n, src, dst, _randint(gen, 1, whi + 1, src.numel())


def _edges(case, seed):
    if case["family"] == "rmat":
        return _rmat(case["n"], seed)
    if case["family"] == "er":
        return _er(case["n"], case["m"], seed)
    return _grid(case["side"], case["whi"], seed)


def _sources(n, src, k, seed):
    """k vertices with out-edges, uniform."""
    has = torch.zeros(n, dtype=torch.bool, device="cuda")
    has[src.long()] = True
    nz = has.nonzero().view(-1)
    at = torch.randint(0, nz.numel(), (k,), generator=_gen(seed), device="cuda")
    return [int(x) for x in nz[at].cpu()]


def _batch_graphs(case):
    """Alternating R-MAT and grid graphs whose sizes spread from 2^lo to 2^hi vertices, none a round number."""
    out = []
    last = max(1, case["graphs"] - 1)
    for i in range(case["graphs"]):
        n = int(2.0 ** (case["lo"] + (case["hi"] - case["lo"]) * i / last))
        if i % 2:
            out.append({"family": "rmat", "n": n - 3 * i})
        else:
            out.append({"family": "grid", "side": math.isqrt(4 * n) - i, "whi": 1000})
    return out


class _Graph:
    """A graph handle that frees its graph when the program drops it."""

    def __init__(self, n, src, dst, w):
        st, self.handle = fg.fg_graph_create_coo(n, src, dst, w)
        fg.check(st)
        self.n = n

    def __del__(self):
        if getattr(self, "handle", None) is not None:
            fg.fg_graph_destroy(self.handle)
            self.handle = None


def _out(n):
    return torch.empty(n, dtype=torch.int32, device="cuda")


def _csr(n, src, dst, w):
    order = torch.sort(src, stable=True).indices
    row = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row[1:] = torch.bincount(src, minlength=n).cumsum(0)
    return row, dst[order].contiguous(), w[order].contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        graphs, queries, outs = [], [], []
        for i, spec in enumerate(_batch_graphs(case)):
            n, src, dst, w = _edges(spec, seed + 1000 * i)
            g = _Graph(n, src, dst, w)
            graphs.append(g)
            outs.append(torch.empty((case["per_graph"], n), dtype=torch.int32, device="cuda"))
            for j, s in enumerate(_sources(n, src, case["per_graph"], seed + 1000 * i + 1)):
                queries.append((g.handle, j % 2, s, outs[i][j], fg.FG_AUTO))
        return {"kind": kind, "graphs": graphs, "queries": queries, "outs": outs}
    n, src, dst, w = _edges(case, seed)
    if kind == "load":
        arrays = (src, dst, w) if case["form"] == "coo" else _csr(n, src, dst, w)
        return {"kind": kind, "form": case["form"], "n": n, "arrays": arrays, "out": _out(n)}
    k = case.get("k", 1)
    return {"kind": kind, "graph": _Graph(n, src, dst, w), "algo": case["algo"], "mode": MODE.get(case.get("mode")),
            "sources": _sources(n, src, k, seed + 1), "outs": [_out(n) for _ in range(k)]}


def run(state):
    kind = state["kind"]
    if kind == "batch":
        st, _, _, _ = fg.fg_run_batch(state["queries"], use_cuda_graph=True, fuse_same_graph=True)
        fg.check(st)
        return state["outs"]
    if kind == "load":
        create = fg.fg_graph_create_coo if state["form"] == "coo" else fg.fg_graph_create_csr
        st, h = create(state["n"], *state["arrays"])
        fg.check(st)
        fg.check(fg.fg_cc(h, state["out"]))
        fg.check(fg.fg_graph_destroy(h))
        return state["out"]
    h, outs = state["graph"].handle, state["outs"]
    if kind == "multi":
        st, _, _ = fg.fg_run_multi(h, ALGO[state["algo"]], state["sources"], outs)
        fg.check(st)
        return outs
    if state["algo"] == "sssp":
        fg.check(fg.fg_sssp(h, state["sources"][0], outs[0], state["mode"]))
    elif state["algo"] == "bfs":
        fg.check(fg.fg_bfs(h, state["sources"][0], outs[0], state["mode"]))
    else:
        fg.check(fg.fg_cc(h, outs[0], state["mode"]))
    return outs[0]


# ---------------------------------------------------------------- what a pass cannot do without
def _size(spec):
    if spec["family"] == "rmat":
        return spec["n"], 16 * spec["n"]
    if spec["family"] == "er":
        return spec["n"], spec["m"]
    side = spec["side"]
    pairs = 2 * side * (side - 1)
    return side * side, 2 * (int(0.98 * pairs) + int(round(0.001 * pairs)))


def work(case):
    """Bytes: the offsets and targets (and, for SSSP, the weights) read once, each output written once; a
    load reads its edge list.  Operations: one addition and one comparison an edge and source."""
    if case["kind"] == "batch":
        total = {"bytes": 0, "flops": 0}
        for spec in _batch_graphs(case):
            n, m = _size(spec)
            total["bytes"] += 4 * n + 8 * m + 4 * n * case["per_graph"]
            total["flops"] += 2 * m * case["per_graph"]
        return total
    n, m = _size(case)
    if case["kind"] == "load":
        return {"bytes": 12 * m + 4 * n, "flops": 2 * m}
    k = case.get("k", 1)
    per_edge = 8 if case["algo"] == "sssp" else 4
    return {"bytes": 4 * n + per_edge * m + 4 * n * k, "flops": 2 * m * k}


# ---------------------------------------------------------------- the same results in plain torch, 64 bits
def _relax(n, src, dst, w, s):
    d = torch.full((n,), INF, dtype=torch.int64, device="cuda")
    d[s] = 0
    while True:
        new = d.clone()
        cand = d[src]
        cand = torch.where(cand == INF, cand, cand + w)
        new.scatter_reduce_(0, dst, cand, "amin")
        if torch.equal(new, d):
            return d
        d = new


def _components(n, src, dst):
    lab = torch.arange(n, dtype=torch.int64, device="cuda")
    while True:
        new = lab.clone()
        new.scatter_reduce_(0, dst, lab[src], "amin")
        new.scatter_reduce_(0, src, lab[dst], "amin")
        while True:
            jumped = new[new]
            if torch.equal(jumped, new):
                break
            new = jumped
        if torch.equal(new, lab):
            return lab
        lab = new


def exact(case, seed):
    if case["kind"] == "batch":
        out = []
        for i, spec in enumerate(_batch_graphs(case)):
            n, src, dst, w = _edges(spec, seed + 1000 * i)
            srcs = _sources(n, src, case["per_graph"], seed + 1000 * i + 1)
            src, dst, w = src.long(), dst.long(), w.long()
            out.append(torch.stack([_relax(n, src, dst, 1 if j % 2 else w, s) for j, s in enumerate(srcs)]))
        return out
    n, src, dst, w = _edges(case, seed)
    if case["kind"] == "load":
        return _components(n, src.long(), dst.long())
    srcs = _sources(n, src, case.get("k", 1), seed + 1)
    src, dst = src.long(), dst.long()
    if case["algo"] == "cc":
        return _components(n, src, dst)
    w = w.long() if case["algo"] == "sssp" else 1
    outs = [_relax(n, src, dst, w, s) for s in srcs]
    return outs if case["kind"] == "multi" else outs[0]
