"""The workloads whose speed this framework answers for: graphs of its users' kinds and sizes through
the public entry points of `paper_2312_04876_gb300`, from one small call to the largest runs.

Graphs are drawn on the GPU from a seed: R-MAT (social and web graphs: hubs, small diameter), planted
partitions (community benchmarks) and road-like grids (low degree, many passes).  Integer weights are
1..8 or 1; float weights are multiples of 1/8 where a whole run returns its membership (their fp32
sums are exact, so the run is reproducible) and arbitrary in the single-step case.
"""
import math

import numpy as np
import torch

import paper_2312_04876_gb300 as lv

DEV = "cuda:0"


# ------------------------------------------------------------------ cases
def listed():
    return [
        # one small graph with the default parameters (deterministic, input checked): an interactive
        # call or the inner step of a larger program, where latency is all
        dict(name="small_default", kind="run", graph="sbm", n=2000, blocks=20, deg=14.0, out=0.3, weights="unit",
             mode="deterministic", validate=1),
        # the 10,000-vertex planted partition in fast mode: the smallest benchmark workload
        dict(name="sbm10k_fast", kind="run", graph="sbm", n=10000, blocks=100, deg=14.9, out=0.33, weights="unit",
             mode="fast", validate=0),
        # a medium planted partition with float weights (similarities), odd sizes, default parameters
        dict(name="sbm100k_fp32", kind="run", graph="sbm", n=100003, blocks=37, deg=25.0, out=0.1, weights="eighths",
             mode="deterministic", validate=1),
        # a social-network graph of ordinary size, deterministic
        dict(name="rmat20_det", kind="run", graph="rmat", scale=20, factor=16, weights="int8", mode="deterministic",
             validate=1),
        # the benchmark's graph, deterministic: the largest single reproducible run
        dict(name="rmat22_det", kind="run", graph="rmat", scale=22, factor=16, weights="int8", mode="deterministic",
             validate=0),
        # the benchmark's graph in fast mode.  The asynchronous schedule is random, so programs run it
        # under several seeds and keep the best: one pass is eight such runs
        dict(name="rmat22_fast_x8", kind="restarts", graph="rmat", scale=22, factor=16, weights="int8", seeds=8),
        # the road-like grid of 24 million vertices, deterministic: rows of 2-5 arcs, many passes
        dict(name="grid24m_det", kind="run", graph="grid", side=4899, weights="unit", mode="deterministic",
             validate=0),
        # many small independent graphs in one call (ego networks, molecules, per-user graphs)
        dict(name="batch_sbm512", kind="batch", graphs=512, n_lo=1000, n_hi=30000, mode="fast"),
        # graph in pinned host memory in, membership on the host out: upload and download included
        dict(name="host_rmat18", kind="host", graph="rmat", scale=18, factor=16, weights="int8",
             mode="deterministic", validate=1),
        # a changing graph: half a percent of the edges deleted, as many inserted, then a warm start
        # from the membership of the graph before
        dict(name="dynamic_rmat20", kind="dynamic", graph="rmat", scale=20, factor=16, weights="int8", share=0.005),
        # a server's burst: mixed requests from host memory through four lanes
        dict(name="serve_mixed", kind="serve", requests=24, e_lo=10000, e_hi=2000000),
        # the single steps on float weights: the modularity of a given membership and the coupling matrix
        # of its communities (one aggregation)
        dict(name="steps_fp32", kind="steps", graph="rmat", scale=20, factor=16, weights="float", comms=1500),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, big):
    """Graph fields of a drawn case; `big`: at most about that many arcs."""
    g = rng.choice(("sbm", "rmat", "grid"))
    if g == "sbm":
        n = _logint(rng, 500, max(1000, min(1500000, big // 20)))
        return dict(graph="sbm", n=n, blocks=max(2, min(n // 20, _logint(rng, 2, 400))),
                    deg=round(rng.uniform(6.0, 40.0), 2), out=round(rng.uniform(0.05, 0.4), 3))
    if g == "rmat":
        top = max(11, min(21, int(math.log2(big / 32))))
        return dict(graph="rmat", scale=rng.randint(10, top), factor=rng.choice((6, 11, 16, 23)))
    return dict(graph="grid", side=_logint(rng, 20, max(40, min(4000, int(math.sqrt(big / 4))))))


def draw(rng):
    kind = rng.choice(("run", "run", "run", "run", "host", "dynamic", "batch", "restarts", "serve", "steps"))
    if kind == "run":
        c = dict(kind=kind, **_draw_graph(rng, 6e7))
        c["weights"] = rng.choice(("unit", "int8", "eighths"))
        # fast mode is reproducible where it takes the colour-synchronous schedule
        small = c["graph"] != "rmat" and (c["n"] if c["graph"] == "sbm" else c["side"] ** 2) < 150000
        c["mode"] = rng.choice(("fast", "deterministic")) if small else "deterministic"
        c["validate"] = rng.randint(0, 1)
        return c
    if kind == "host":
        return dict(kind=kind, **_draw_graph(rng, 1.5e7), weights=rng.choice(("unit", "int8")), mode="deterministic",
                    validate=rng.randint(0, 1))
    if kind == "dynamic":
        return dict(kind=kind, **_draw_graph(rng, 3e7), weights="int8", share=round(rng.uniform(0.0005, 0.02), 5))
    if kind == "batch":
        lo = _logint(rng, 200, 3000)
        return dict(kind=kind, graphs=_logint(rng, 8, 400), n_lo=lo, n_hi=lo * rng.randint(2, 10),
                    mode=rng.choice(("fast", "deterministic")))
    if kind == "restarts":
        return dict(kind=kind, graph="rmat", scale=rng.randint(18, 21), factor=rng.choice((11, 16)), weights="int8",
                    seeds=8)
    if kind == "serve":
        return dict(kind=kind, requests=rng.randint(5, 30), e_lo=_logint(rng, 2000, 20000),
                    e_hi=_logint(rng, 100000, 2000000))
    return dict(kind=kind, **_draw_graph(rng, 3e7), weights=rng.choice(("float", "int8")),
                comms=_logint(rng, 20, 2000))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _rand(g, k, dtype=torch.float32):
    return torch.rand(k, generator=g, device=DEV, dtype=dtype)


def _below(g, k, hi):
    return torch.randint(0, hi, (k,), generator=g, device=DEV)


def _pairs_rmat(g, scale, factor):
    """Undirected R-MAT draws (0.57, 0.19, 0.19, 0.05) as keys lo << 32 | hi."""
    total, keys = factor << scale, []
    for d0 in range(0, total, 1 << 25):
        k = min(1 << 25, total - d0)
        u = torch.zeros(k, dtype=torch.int32, device=DEV)
        v = torch.zeros(k, dtype=torch.int32, device=DEV)
        for _ in range(scale):
            r = _rand(g, k)
            ub = r >= 0.76
            vb = ((r >= 0.57) & (r < 0.76)) | (r >= 0.95)
            u = u * 2 + ub.to(torch.int32)
            v = v * 2 + vb.to(torch.int32)
        keys.append(_keys(u.to(torch.int64), v.to(torch.int64)))
    return torch.cat(keys)


def _keys(u, v):
    keep = u != v
    u, v = u[keep], v[keep]
    return (torch.minimum(u, v) << 32) | torch.maximum(u, v)


def _pairs_sbm(g, n, blocks, deg, out):
    """Planted partition: n * deg / 2 draws, a share `out` of them between any two vertices."""
    m = int(n * deg / 2)
    u = _below(g, m, n)
    b = u * blocks // n
    lo = (b * n + blocks - 1) // blocks
    hi = ((b + 1) * n + blocks - 1) // blocks
    inside = lo + (_rand(g, m, torch.float64) * (hi - lo)).to(torch.int64)
    v = torch.where(_rand(g, m) < out, _below(g, m, n), torch.minimum(inside, hi - 1))
    return _keys(u, v)


def _pairs_grid(g, side):
    """Road-like lattice: 10% of the edges deleted, 1% random long links."""
    n = side * side
    at = torch.arange(n, device=DEV)
    right, down = at[at % side != side - 1], at[: n - side]
    u = torch.cat([right, down])
    v = torch.cat([right + 1, down + side])
    keep = _rand(g, u.numel()) >= 0.1
    u, v = u[keep], v[keep]
    k = u.numel() // 100
    return torch.cat([_keys(u, v), _keys(_below(g, k, n), _below(g, k, n))])


def _vertices(c):
    return {"rmat": lambda: 1 << c["scale"], "sbm": lambda: c["n"], "grid": lambda: c["side"] ** 2}[c["graph"]]()


def _edges(c, g):
    if c["graph"] == "rmat":
        return _pairs_rmat(g, c["scale"], c["factor"])
    if c["graph"] == "sbm":
        return _pairs_sbm(g, c["n"], c["blocks"], c["deg"], c["out"])
    return _pairs_grid(g, c["side"])


def _weights(g, k, what):
    if what == "unit":
        return torch.ones(k, dtype=torch.int32, device=DEV)
    if what == "int8":
        return _below(g, k, 8).to(torch.int32) + 1
    if what == "eighths":
        return (_below(g, k, 8).to(torch.float32) + 1) / 8
    return 1.0 - _rand(g, k)


def _csr(keys, n, g, weights):
    """Symmetric CSR (offsets int64, targets int32, weights) of undirected edge keys, rows by target."""
    e = torch.unique(keys)
    w = _weights(g, e.numel(), weights)
    lo, hi = e >> 32, e & 0xFFFFFFFF
    both, order = torch.sort(torch.cat([e, (hi << 32) | lo]))
    offsets = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(both >> 32, minlength=n), 0, out=offsets[1:])
    return offsets, (both & 0xFFFFFFFF).to(torch.int32), torch.cat([w, w])[order]


def _graph(c, seed):
    g = _gen(seed)
    return _csr(_edges(c, g), _vertices(c), g, c["weights"])


def _request(g, edges, odd):
    """One served graph of about `edges` edges as host arrays."""
    if odd:
        scale = max(8, int(math.ceil(math.log2(edges / 16))))
        c = dict(graph="rmat", scale=scale, factor=max(1, round(edges / (1 << scale))))
    else:
        n = max(100, edges // 8)
        c = dict(graph="sbm", n=n, blocks=2 + n % 31, deg=16.0, out=0.1)
    o, t, w = _csr(_edges(c, g), _vertices(c), g, "int8")
    return o.cpu().numpy(), t.cpu().numpy(), w.cpu().numpy()


def _spread(c, key_lo, key_hi, count):
    """`count` sizes spread over [lo, hi] by their logarithm."""
    lo, hi = math.log(c[key_lo]), math.log(c[key_hi])
    return [int(round(math.exp(lo + (hi - lo) * ((k * 0.6180339887498949) % 1.0)))) for k in range(count)]


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        # the graphs of a batch as one segmented CSR with graph-local targets
        sizes = _spread(c, "n_lo", "n_hi", c["graphs"])
        vo = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        offs, tgs, ws, base = [torch.zeros(1, dtype=torch.int64, device=DEV)], [], [], 0
        for k, n in enumerate(sizes):
            g = _gen(seed * 100003 + k)
            o, t, w = _csr(_pairs_sbm(g, n, 2 + k % 63, 4.0 + 60.0 * ((k * 0.7548776662466927) % 1.0), 0.02 + 0.1 * (k % 3)),
                           n, g, "unit")
            offs.append(o[1:] + base)
            base += t.numel()
            tgs.append(t)
            ws.append(w)
        return dict(c=c, handle=lv.Louvain(0), vo=vo, graph=(torch.cat(offs), torch.cat(tgs), torch.cat(ws)))
    if c["kind"] == "serve":
        sizes = _spread(c, "e_lo", "e_hi", c["requests"])
        server = lv.Server(device=0, hbm_budget_bytes=16 << 30, lanes=4, mode="deterministic", validate=0)
        return dict(c=c, server=server,
                    graphs=[_request(_gen(seed * 1009 + k), e, k % 2 == 1) for k, e in enumerate(sizes)])
    s = dict(c=c, handle=lv.Louvain(0), graph=_graph(c, seed))
    if c["kind"] == "host":
        s["graph"] = tuple(x.cpu().pin_memory() for x in s["graph"])
    elif c["kind"] == "steps":
        n = _vertices(c)
        nc = max(1, min(c["comms"], n))
        s["nc"] = nc
        # skewed community sizes, every id used
        m = (_rand(_gen(seed + 1), n, torch.float64) ** 2 * nc).to(torch.int32).clamp_(max=nc - 1)
        m[:nc] = torch.arange(nc, dtype=torch.int32, device=DEV)
        s["membership"] = m
    elif c["kind"] == "dynamic":
        o, t, w = s["graph"]
        n, g = o.numel() - 1, _gen(seed + 1)
        k = max(1, int(t.numel() / 2 * c["share"]))
        at = _below(g, k, t.numel())
        rows = torch.searchsorted(o, at, right=True) - 1
        s["delete"] = torch.stack([rows.to(torch.int32), t[at]], 1)
        s["insert"] = torch.stack([_below(g, k, n), _below(g, k, n)], 1).to(torch.int32)
        s["insert_w"] = _weights(g, k, c["weights"])
        s["before"], _ = s["handle"].run(o, t, w, mode="deterministic", validate=0)
    return s


# ------------------------------------------------------------------ the pass
def run(state):
    c = state["c"]
    if c["kind"] == "serve":
        server = state["server"]
        tickets = [server.submit(*g) for g in state["graphs"]]
        got = [server.result(t) for t in tickets]
        return [np.concatenate([m for m, _ in got]), np.array([i["modularity"] for _, i in got])]
    h = state["handle"]
    if c["kind"] == "batch":
        m, graphs, _ = h.run_batch(state["vo"], *state["graph"], mode=c["mode"], validate=0)
        return [m, np.array([r["modularity"] for r in graphs]), np.array([r["passes"] for r in graphs])]
    o, t, w = state["graph"]
    if c["kind"] == "run":
        m, r = h.run(o, t, w, mode=c["mode"], validate=c["validate"])
        return [m, r.modularity, r.passes, r.total_iterations]
    if c["kind"] == "host":
        m, r = h.run_host(o, t, w, mode=c["mode"], validate=c["validate"])
        return [m, r.modularity, r.passes, r.total_iterations]
    if c["kind"] == "restarts":
        return np.array([h.run(o, t, w, mode="fast", validate=0, seed=s)[1].modularity for s in range(c["seeds"])])
    if c["kind"] == "dynamic":
        o2, t2, w2 = h.update_graph(o, t, w, o.numel() - 1, state["delete"], state["insert"], state["insert_w"])
        m, r = h.run_from(o2, t2, w2, state["before"], mode="deterministic", validate=0)
        return [o2, m, r.modularity, r.passes, r.total_iterations]
    # steps: the super-vertex graph as a dense matrix (its rows come unordered)
    nc = state["nc"]
    q = h.modularity(o, t, w, state["membership"])
    o2, t2, w2 = h.aggregate(o, t, w, state["membership"], nc)
    rows = torch.repeat_interleave(torch.arange(nc, device=DEV), o2[1:] - o2[:-1], output_size=t2.numel())
    matrix = torch.zeros(nc * nc, dtype=w2.dtype, device=DEV)
    matrix[rows * nc + t2] = w2
    return [q, o2, matrix]


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    c = dict(case)
    if c["kind"] == "serve":
        e = sum(_spread(c, "e_lo", "e_hi", c["requests"]))
        return {"bytes": 16.0 * e + 12.0 * e / 8, "flops": 4.0 * e}
    if c["kind"] == "batch":
        sizes = _spread(c, "n_lo", "n_hi", c["graphs"])
        a = sum(n * (4.0 + 60.0 * ((k * 0.7548776662466927) % 1.0)) for k, n in enumerate(sizes))
        return {"bytes": 8.0 * a + 12.0 * sum(sizes), "flops": 2.0 * a}
    n = _vertices(c)
    # arcs kept after deduplication, about
    a = {"rmat": lambda: 1.9 * c["factor"] * n, "sbm": lambda: n * c["deg"], "grid": lambda: 3.6 * n}[c["graph"]]()
    times = c.get("seeds", 1)
    b = 8.0 * a + 12.0 * n
    if c["kind"] == "dynamic":
        b = 2 * b + 8.0 * a  # the old graph read, the new one written and read
    return {"bytes": times * b, "flops": times * 2.0 * a}


# ------------------------------------------------------------------ 64-bit values
def exact(case, seed):
    c = dict(case)
    if c["kind"] != "steps":
        return None  # a run's modularity is that of the membership it finds, which has no closed form
    o, t, w = _graph(c, seed)
    n = o.numel() - 1
    nc = max(1, min(c["comms"], n))
    m = (_rand(_gen(seed + 1), n, torch.float64) ** 2 * nc).to(torch.int32).clamp_(max=nc - 1)
    m[:nc] = torch.arange(nc, dtype=torch.int32, device=DEV)
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), o[1:] - o[:-1])
    key = m[rows].to(torch.int64) * nc + m[t.to(torch.int64)].to(torch.int64)
    w = w.to(torch.float64)
    matrix = torch.zeros(nc * nc, dtype=torch.float64, device=DEV).index_add_(0, key, w)
    two_m, square = w.sum(), matrix.view(nc, nc)
    q = float(square.diagonal().sum() / two_m - (square.sum(1) / two_m).square().sum())
    return [q, None, matrix]
