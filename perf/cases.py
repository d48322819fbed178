"""The work that a user of this framework has it do, as cases that can be timed.

Every case is one pass through the public binding (``mscd.Context``): a run
over every seed and scale of a graph, one share of a larger run's seeds, a
batch of graphs, queries to the server, growth into the caller's own buffers,
growth from given communities, the full method, the NMI of two covers, a graph
load.  Sizes are those of the benchmark's workloads (planted-1k, lfr-100k, the
weighted 1M-node graph, the uneven batch, the 2M-node serving graphs, the
accuracy study), with the seeds thinned where all of them would take long; the
graphs are drawn on the GPU from the seed.
"""
import ctypes
import math
import random

import numpy as np
import torch

from paper_1301_0955_gb300 import mscd

DEV = "cuda:0"


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest job: all 1,000 nodes of the planted partition at 8 scales (launches and
        # host steps count as much as growth)
        dict(name="run planted 1k", kind="run", graph="planted", n=1000, deg=22, weighted=False, scales=8,
             lo=0.5, hi=1.0, share=1, parts=1),
        # the accuracy study's graph: 10,000 nodes in communities of 10-50, 40 scales from 0.3;
        # every second node a seed
        dict(name="run accuracy 10k", kind="run", graph="small-comms", n=10000, deg=19, weighted=False, scales=40,
             lo=0.3, hi=1.0, share=2, parts=1),
        # lfr-100k at its 20 scales: the share of one of 8 GPUs (every 8th node a seed)
        dict(name="run lfr-100k 1 of 8", kind="run", graph="lfr", n=100000, deg=20, weighted=False, scales=20,
             lo=0.5, hi=1.0, share=8, parts=1),
        # the weighted 1M-node graph at its 32 scales, every 80th node a seed
        dict(name="run lfr-1m weighted 1 of 80", kind="run", graph="lfr3", n=1000000, deg=30, weighted=True,
             scales=32, lo=0.5, hi=1.0, share=80, parts=1),
        # many graphs in one call: 12 graphs of log-uniform sizes as one union, 16 scales, every
        # second node a seed
        dict(name="run union of 12", kind="run", graph="lfr", n=10000, deg=25, weighted=False, scales=16, lo=0.5,
             hi=1.0, share=2, parts=12),
        # growth from given communities (initial members) on a weighted graph
        dict(name="run_init 50k weighted", kind="init", graph="lfr", n=50000, deg=20, weighted=True, scales=6,
             lo=0.5, hi=1.0, share=0, parts=1),
        # the server: one seed's community, the latency of a single query on a 2M-node graph
        dict(name="serve 1 seed", kind="serve", graph="lfr3", n=2000000, deg=25, weighted=False, scales=16, lo=0.5,
             hi=1.0, queries=1, max_seeds=1),
        # the server: 16 queries of 1-4096 seeds at mixed scales arriving together
        dict(name="serve 16 queries", kind="serve", graph="lfr3", n=2000000, deg=25, weighted=False, scales=16,
             lo=0.5, hi=1.0, queries=16, max_seeds=4096),
        # growth into the caller's buffers without device allocation, at the fine scales
        dict(name="grow_noalloc 100k", kind="noalloc", graph="lfr", n=100000, deg=20, weighted=False, scales=4,
             lo=0.8, hi=1.0, seeds=2048),
        # the paper's whole Alg. 2 with seed rule 1
        dict(name="full method 30k", kind="full", graph="lfr", n=30000, deg=20, weighted=False, scales=8, lo=0.5,
             hi=1.0, rule=1),
        # the NMI of two covers of 100,000 nodes with overlapping communities
        dict(name="nmi of covers 100k", kind="nmi", n=100000, copies=8),
        # a weighted graph's load from device arrays (checks, exact weights, degrees)
        dict(name="load 1m weighted", kind="load", graph="lfr3", n=1000000, deg=30, weighted=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "init", "serve", "serve", "noalloc", "full", "nmi", "load"])
    weighted = rng.random() < 0.4
    deg = rng.randint(10, 40)
    lo = round(rng.uniform(0.5, 0.8), 3)
    if kind == "run":
        parts = rng.choice([1, 1, 1, rng.randint(2, 12)])
        graph = rng.choice(["lfr", "lfr", "lfr3", "small-comms", "planted"]) if parts == 1 else "lfr"
        if graph == "planted":
            return dict(kind="run", graph="planted", n=50 * rng.randint(4, 40), deg=22, weighted=weighted,
                        scales=rng.randint(2, 12), lo=lo, hi=1.0, share=1, parts=1)
        if graph == "small-comms":
            lo = round(rng.uniform(0.3, 0.8), 3)
        n = _log(rng, 2000, 1000000) if parts == 1 else _log(rng, 2000, 12000)
        units = _log(rng, 10000, 200000)
        scales = rng.randint(4, 32)
        share = max(1, n * scales // units if parts == 1 else n * parts * scales // (2 * units))
        return dict(kind="run", graph=graph, n=n, deg=deg, weighted=weighted, scales=scales, lo=lo, hi=1.0,
                    share=share, parts=parts)
    if kind == "init":
        return dict(kind="init", graph="lfr", n=_log(rng, 5000, 100000), deg=deg, weighted=weighted,
                    scales=rng.randint(2, 8), lo=lo, hi=1.0, share=0, parts=1)
    if kind == "serve":
        return dict(kind="serve", graph="lfr3", n=_log(rng, 200000, 2000000), deg=min(deg, 25), weighted=weighted,
                    scales=16, lo=0.5, hi=1.0, queries=rng.randint(1, 16), max_seeds=_log(rng, 1, 4096))
    if kind == "noalloc":
        return dict(kind="noalloc", graph="lfr", n=_log(rng, 2000, 200000), deg=min(deg, 25), weighted=weighted,
                    scales=rng.randint(1, 6), lo=0.85, hi=1.0, seeds=_log(rng, 1, 2048))
    if kind == "full":
        return dict(kind="full", graph="lfr", n=_log(rng, 2000, 30000), deg=min(deg, 25), weighted=weighted,
                    scales=rng.randint(3, 8), lo=0.5, hi=1.0, rule=rng.choice([1, 2]))
    if kind == "nmi":
        return dict(kind="nmi", n=_log(rng, 2000, 100000), copies=rng.randint(1, 8))
    return dict(kind="load", graph=rng.choice(["lfr", "lfr3"]), n=_log(rng, 10000, 1000000), deg=deg,
                weighted=weighted)


# ---------------------------------------------------------------- graphs
def _powerlaw(lo, hi, tau, count, g):
    ks = torch.arange(lo, hi + 1, dtype=torch.float64, device=DEV)
    cdf = torch.cumsum(ks ** -tau, 0)
    x = torch.rand(count, generator=g, device=DEV, dtype=torch.float64) * cdf[-1]
    return lo + torch.searchsorted(cdf, x).clamp_(max=hi - lo)


def _kmin(mean, kmax, tau):
    best, err = 1, None
    for k in range(1, kmax + 1):
        ks = np.arange(k, kmax + 1, dtype=np.float64)
        p = ks ** -tau
        e = abs((ks * p).sum() / p.sum() - mean)
        if err is None or e < err:
            best, err = k, e
    return best


def _pairs(stub_node, stub_group, g):
    """Stubs paired at random inside their group (configuration model)."""
    order = torch.argsort(torch.rand(stub_node.numel(), generator=g, device=DEV), stable=True)
    order = order[torch.argsort(stub_group[order], stable=True)]
    s, gr = stub_node[order], stub_group[order]
    start = torch.ones_like(gr, dtype=torch.bool)
    start[1:] = gr[1:] != gr[:-1]
    idx = torch.arange(gr.numel(), device=DEV)
    first = torch.cummax(torch.where(start, idx, torch.zeros_like(idx)), 0).values
    lead = ((idx - first) % 2 == 0)
    lead[-1:] = False
    lead[:-1] &= gr[1:] == gr[:-1]
    i = torch.nonzero(lead).reshape(-1)
    return s[i], s[i + 1]


def _csr(n, a, b, weighted, g):
    keep = a != b
    a, b = a[keep], b[keep]
    key = torch.unique(torch.minimum(a, b) * n + torch.maximum(a, b))
    a, b = key // n, key % n
    w = None
    if weighted:  # float32 uniform in [0.5, 2], one per undirected edge
        w = 0.5 + 1.5 * torch.rand(a.numel(), generator=g, device=DEV)
        w = torch.cat([w, w])
    both, order = torch.sort(torch.cat([a * n + b, b * n + a]))
    src = both // n
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return rp, (both % n).to(torch.int32).contiguous(), w[order].contiguous() if weighted else None


_SHAPES = {  # largest degree over the mean, degree and size exponents, community sizes, mixing per level
    "lfr": (10, 2.5, 1.5, (20, 1000), (0.3, 0.1)),
    "lfr3": (10, 2.5, 1.5, (20, 1000), (0.3, 0.2, 0.1)),
    "small-comms": (5, 2.0, 1.0, (10, 50), (0.2, 0.05)),
}


def _graph(shape, n, deg, weighted, g):
    """(row_ptr, col, w or None) on the GPU, and the finest communities."""
    if shape == "planted":
        comm = torch.arange(n, device=DEV) // 50
        sup = comm // 5
        p = torch.where(comm[:, None] == comm[None], 0.3, torch.where(sup[:, None] == sup[None], 0.03, 0.002))
        a, b = torch.nonzero(torch.triu(torch.rand(n, n, generator=g, device=DEV) < p, 1), as_tuple=True)
        return _csr(n, a, b, weighted, g) + (comm,)
    spread, tau, tau_s, (smin, smax), mixing = _SHAPES[shape]
    kmax = spread * deg
    k = _powerlaw(_kmin(deg, kmax, tau), kmax, tau, n, g)
    # micro communities of power-law sizes, grouped by 2-6 into each next level
    sizes = _powerlaw(smin, smax, tau_s, n // smin + 1, g)
    ends = torch.cumsum(sizes, 0)
    label = torch.searchsorted(ends, torch.arange(n, device=DEV), right=True)
    label = label[torch.randperm(n, generator=g, device=DEV)]
    micro, us, vs = label, [], []
    node = torch.arange(n, device=DEV)
    left = k.clone()
    for level, mu in enumerate(mixing + (0.0,)):
        inner = (k.double() * (1.0 - mu)).round().long() - (k - left)
        if level == 0:
            inner = torch.minimum(inner, sizes[micro] - 1)
        inner = torch.minimum(inner.clamp_(min=0), left)
        stubs = torch.repeat_interleave(node, inner)
        group = label if level < len(mixing) else torch.zeros_like(label)
        a, b = _pairs(stubs, group[stubs], g)
        us.append(a)
        vs.append(b)
        left = left - inner
        m = int(label.max()) + 1
        up = torch.cumsum(torch.randint(2, 7, (m,), generator=g, device=DEV), 0)
        label = torch.searchsorted(up, torch.randperm(m, generator=g, device=DEV), right=True)[label]
    return _csr(n, torch.cat(us), torch.cat(vs), weighted, g) + (micro,)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


# room for the entries of a unit's list in the caller's arrays
_ROOM = {"lfr": 384, "lfr3": 384, "small-comms": 384, "planted": 1000}


def _part_sizes(case):
    r = random.Random(case["parts"])
    return [_log(r, 1000, case["n"]) for _ in range(case["parts"])]


def _cover(n, copies, g, base):
    """Overlapping communities: `copies` versions of every base community, each
    without some of its members and with a few others."""
    node = torch.arange(n, device=DEV)
    keys = []
    for c in range(copies):
        stay = torch.rand(n, generator=g, device=DEV) < 0.95
        move = torch.randint(0, n, (n // 20,), generator=g, device=DEV)
        comm = torch.cat([base[stay], base[torch.randint(0, n, (n // 20,), generator=g, device=DEV)]])
        keys.append((comm * copies + c) * n + torch.cat([node[stay], move]))
    key = torch.unique(torch.cat(keys))
    comm, nodes = key // n, key % n
    counts = torch.unique_consecutive(comm, return_counts=True)[1]
    ptr = np.zeros(counts.numel() + 1, np.int64)
    ptr[1:] = np.cumsum(counts.cpu().numpy())
    return ptr, nodes.to(torch.int32).cpu().numpy()


def prepare(case, seed):
    g = _gen(seed)
    kind, n = case["kind"], case["n"]
    ctx = mscd.Context(0)
    st = dict(kind=kind, ctx=ctx, n=n)
    if kind == "nmi":
        sizes = _powerlaw(20, 1000, 1.5, n // 20 + 1, g)
        base = torch.searchsorted(torch.cumsum(sizes, 0), torch.arange(n, device=DEV), right=True)
        base = base[torch.randperm(n, generator=g, device=DEV)]
        st["a"] = _cover(n, case["copies"], g, base)
        st["b"] = _cover(n, case["copies"], g, base)
        return st
    if kind == "run" and case["parts"] > 1:
        sizes = _part_sizes(case)
        ids = [ctx.load_csr(m, *_graph(case["graph"], m, case["deg"], case["weighted"], g)[:3]) for m in sizes]
        st["gid"] = ctx.graph_union(ids)
        n = sum(sizes)
    else:
        rp, col, w, micro = _graph(case["graph"], n, case["deg"], case["weighted"], g)
        if kind == "load":
            st.update(rp=rp, col=col, w=w)
            torch.cuda.synchronize()
            return st
        torch.cuda.synchronize()
        st["gid"] = ctx.load_csr(n, rp, col, w)
    st["alphas"] = mscd.scales_logspaced(case["lo"], case["hi"], case["scales"])
    S, L = case["scales"], _ROOM[case["graph"]]
    if kind in ("run", "init"):
        if kind == "run":
            st["seeds"] = np.arange(seed % case["share"], n, case["share"], dtype=np.int32)[:n // case["share"]]
        else:
            # a part of the micro communities: the first node is the seed, half of the others are given
            m = micro.cpu().numpy()
            order = np.argsort(m, kind="stable")
            order = order[:np.searchsorted(m[order], n // 300)]
            first = np.r_[True, m[order][1:] != m[order][:-1]]
            st["seeds"] = order[first].astype(np.int32)[:n // 300]
            keep = ~first & (np.random.default_rng(seed).random(len(order)) < 0.5)
            given = np.bincount((np.cumsum(first) - 1)[keep], minlength=int(first.sum()))
            st["init_ptr"] = np.r_[0, np.cumsum(given)].astype(np.int64)
            st["init_nodes"] = order[keep].astype(np.int32)
        N = st["units"] = len(st["seeds"])
        if kind == "run" and case["share"] == 1:
            st["seeds"] = None  # every node
        st["host"] = dict(ptr=np.zeros(S * (N + 1), np.int64), nodes=np.zeros(S * N * L, np.int32),
                          fitness=np.zeros(S * N), seed2comm=np.zeros(S * N, np.int32), count=np.zeros(S, np.int64))
    elif kind == "serve":
        r = np.random.default_rng(seed)
        sizes = random.Random(case["queries"] * case["max_seeds"])
        st["queries"], st["host"] = [], []
        for i in range(case["queries"]):
            m = min(n, sizes.randint(1, case["max_seeds"]))
            s = np.unique(r.integers(0, n, 2 * m + 8)).astype(np.int32)
            st["queries"].append((r.permutation(s)[:m], float(st["alphas"][sizes.randrange(S)])))
            st["host"].append((np.zeros(m + 1, np.int64), np.zeros(m * 1024 + 65536, np.int32), np.zeros(m)))
        ctx.serve_start()
    elif kind == "noalloc":
        m = min(n, case["seeds"])
        st["seeds"] = torch.randperm(n, generator=g, device=DEV)[:m].to(torch.int32).contiguous()
        units = m * S
        dev = dict(nodes=(torch.int32, units * 1024 + 8192), offset=(torch.int64, units), len=(torch.int32, units),
                   fitness=(torch.float64, units), stats=(torch.int64, units * mscd.NSTATS),
                   status=(torch.int32, units), hash=(torch.int64, units))
        st["out"] = {k: torch.zeros(c, dtype=t, device=DEV) for k, (t, c) in dev.items()}
        st["lists"] = torch.zeros(units * 1024 + 8192, dtype=torch.int32, device=DEV)
    elif kind == "full":
        st["prio"] = np.random.default_rng(seed).permutation(n).astype(np.int32)
        st["rule"] = case["rule"]
        st["host"] = dict(ptr=np.zeros(S * (n + 1), np.int64), nodes=np.zeros(S * n * 8, np.int32),
                          seeds=np.zeros(S * n, np.int32), fitness=np.zeros(S * n), chosen=np.zeros(n, np.int32),
                          nmi_next=np.zeros(S), count=np.zeros(S + 1, np.int64))
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------- one pass
def _at(a, i=0):
    return a.ctypes.data + i * a.itemsize


def _typed(a, i, t):
    return ctypes.cast(_at(a, i), t)


def _ok(rc):
    if rc not in (mscd.OK, mscd.ETIMEOUT, mscd.EUNDECIDED):
        raise mscd.MscdError(rc)
    return rc


def _communities(st):
    """Every scale's communities, one after the other in the caller's arrays."""
    L, h, b, N = mscd.load(), st["ctx"].h, st["host"], st["units"]
    C, E = ctypes.c_int64(), ctypes.c_int64()
    at, room = 0, len(b["nodes"])
    for s in range(len(st["alphas"])):
        _ok(L.mscd_get_communities(h, s, _typed(b["ptr"], s * (N + 1), mscd.i64p), N + 1,
                                   _typed(b["nodes"], at, mscd.i32p), room - at,
                                   _typed(b["fitness"], s * N, mscd.f64p), _typed(b["seed2comm"], s * N, mscd.i32p),
                                   ctypes.byref(C), ctypes.byref(E)))
        b["count"][s] = C.value
        at += E.value
    return dict(b, stability=st["ctx"].stability())


def run(state):
    ctx, kind = state["ctx"], state["kind"]
    L, i64 = mscd.load(), ctypes.c_int64
    if kind == "run":
        status = ctx.run(state["gid"], state["alphas"], state["seeds"])
        return dict(_communities(state), status=status)
    if kind == "init":
        status = ctx.run_init(state["gid"], state["alphas"], state["seeds"], state["init_ptr"], state["init_nodes"])
        return dict(_communities(state), status=status)
    if kind == "serve":
        ids = [ctx.submit(state["gid"], s, a) for s, a in state["queries"]]
        for q, (ptr, nodes, f) in zip(ids, state["host"]):
            ctx.wait(q)
            _ok(L.mscd_query_result(ctx.h, q, _typed(ptr, 0, mscd.i64p), _typed(nodes, 0, mscd.i32p), len(nodes),
                                    _typed(f, 0, mscd.f64p), ctypes.byref(i64()), None))
        return state["host"]
    if kind == "noalloc":
        o = state["out"]
        status, need = ctx.grow_noalloc(state["gid"], state["alphas"], state["seeds"], o)
        # lists lie in the order the units finished in: read them in the units' order
        end = torch.cumsum(o["len"], 0)
        at = torch.repeat_interleave(o["offset"] - end + o["len"], o["len"], output_size=need)
        state["lists"][:need] = o["nodes"][at + torch.arange(need, device=DEV)]
        return dict(nodes=state["lists"], len=o["len"], fitness=o["fitness"], unit_status=o["status"],
                    hash=o["hash"], status=status)
    if kind == "full":
        b, n = state["host"], state["n"]
        status = ctx.full_run(state["gid"], state["alphas"], prio=state["prio"], seed_rule=state["rule"])
        C, E, at = i64(), i64(), 0
        _ok(L.mscd_full_get_seeds(ctx.h, _typed(b["chosen"], 0, mscd.i32p), n, ctypes.byref(C)))
        b["count"][-1] = C.value
        for s in range(len(state["alphas"])):
            _ok(L.mscd_full_get_scale(ctx.h, s, _typed(b["ptr"], s * (n + 1), mscd.i64p), n + 1,
                                      _typed(b["nodes"], at, mscd.i32p), len(b["nodes"]) - at,
                                      _typed(b["seeds"], s * n, mscd.i32p), _typed(b["fitness"], s * n, mscd.f64p),
                                      ctypes.byref(C), ctypes.byref(E)))
            _ok(L.mscd_full_get_info(ctx.h, s, ctypes.byref(i64()), ctypes.byref(i64()), ctypes.byref(i64()),
                                     _typed(b["nmi_next"], s, mscd.f64p)))
            b["count"][s] = C.value
            at += E.value
        return dict(b, status=status)
    if kind == "nmi":
        return ctx.nmi_covers(state["n"], state["a"], state["b"])
    gid = ctx.load_csr(state["n"], state["rp"], state["col"], state["w"])
    info, k = ctx.graph_info(gid), ctx.graph_degrees(gid)
    ctx.free_graph(gid)
    return dict(degrees=k, **info)


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Bytes: the graph once, and of the results a mean community of 150 nodes
    (30 in small communities) per query seed, and per three seeds of a run,
    whose results are stored once per different community.  Operations: for
    every unit the entries of its members' rows, each a look-up and an update
    (10 operations).  A load reads every entry and its partner's."""
    kind, n = case["kind"], case["n"]
    if kind == "nmi":
        m = n * case["copies"]
        return dict(bytes=8.0 * m, flops=20.0 * m * case["copies"])
    parts = case.get("parts", 1)
    nodes = n if parts == 1 else parts * (n - 1000) / math.log(n / 1000.0 + 1e-9)
    graph = nodes * (8 + case["deg"] * (8 if case["weighted"] else 4))
    if kind == "load":
        return dict(bytes=2.0 * graph + 20 * nodes, flops=10.0 * nodes * case["deg"])
    mean = 30 if case["graph"] == "small-comms" else 100 if case["graph"] == "planted" else 150
    units, each = dict(run=lambda: (nodes / case["share"] * case["scales"] if kind == "run" else 0, 1 / 3),
                       init=lambda: (n / 140 * case["scales"], 1),
                       serve=lambda: (case["queries"] * (case["max_seeds"] + 1) / 2, 1),
                       noalloc=lambda: (case["seeds"] * case["scales"], 1),
                       full=lambda: (nodes / 5, 1 / 3))[kind]()
    rows = units * mean * case["deg"]
    # a few queries need only the rows they meet
    read = min(graph, rows * (8 if case["weighted"] else 4))
    return dict(bytes=read + units * (each * mean * 4 + 12), flops=10.0 * rows)


# ---------------------------------------------------------------- the same in 64 bits
def _grow_dense(A, k, alpha):
    """Every node's community at one scale on a dense adjacency matrix: pop the
    queued node of the largest d/k^alpha (equal ones by id), add it if the
    fitness K/V^alpha rises, else drop it until an addition touches it; then
    remove members in ascending id while that raises the fitness; all again
    while something was added.  Values within 1e-12 are equal."""
    n, tie = len(A), 1e-12
    unit, ids = torch.arange(n, device=DEV), torch.arange(n, device=DEV)
    M = torch.eye(n, dtype=torch.bool, device=DEV)
    D, K, V = A.clone(), torch.zeros(n, dtype=torch.float64, device=DEV), k.clone()
    logk = torch.log(k)
    live = torch.ones(n, dtype=torch.bool, device=DEV)
    inf = float("inf")

    def step(rows, who, sign):
        M[rows, who] = sign > 0
        K[rows] += sign * 2 * D[rows, who]
        V[rows] += sign * k[who]
        D[rows] += sign * A[who]

    while bool(live.any()):
        Q = ~M & (D > 0) & live[:, None]
        added = torch.zeros_like(live)
        while True:
            gain = torch.log1p(2 * D / K[:, None]) - alpha * torch.log1p(k[None] / V[:, None])
            rank = torch.where(Q & ((gain > tie) | (K[:, None] == 0)), torch.log(D) - alpha * logk, -inf)
            top = rank.max(1).values
            rows = torch.nonzero(top > -inf).reshape(-1)
            if not rows.numel():
                break
            who = (rank[rows] >= top[rows, None] - tie).int().argmax(1)
            r = torch.log(D[rows]) - alpha * logk
            t = top[rows, None]
            Q[rows] &= ~((r > t + tie) | ((r >= t - tie) & (ids[None] < who[:, None])))
            step(rows, who, 1)
            Q[rows] = (Q[rows] | (A[who] > 0)) & ~M[rows]
            added[rows] = True
        removing = added.clone()
        while bool(removing.any()):
            last = torch.full((n,), -1, device=DEV)
            some = torch.zeros_like(removing)
            while True:
                left = K[:, None] - 2 * D
                gain = torch.log(left.clamp(min=1e-300) / K[:, None]) - alpha * torch.log1p(-k[None] / V[:, None])
                can = M & (gain > tie) & (left > 0) & (ids[None] > last[:, None]) & removing[:, None]
                can &= ids[None] != unit[:, None]
                rows = torch.nonzero(can.any(1)).reshape(-1)
                if not rows.numel():
                    break
                who = can[rows].int().argmax(1)
                step(rows, who, -1)
                last[rows] = who
                some[rows] = True
            removing = some
        live = added
    f = torch.where(K > 0, torch.exp(torch.log(K) - alpha * torch.log(V)), 0.0)
    return M.cpu().numpy(), f.cpu().numpy()


def _h(x, n):
    p = x / n
    return torch.where(x > 0, -p * torch.log2(p.clamp(min=1e-300)), torch.zeros_like(p))


def _nmi_dense(X, Y, n):
    """Overlapping NMI of two covers given as 0/1 matrices (communities x nodes)."""
    sx, sy = X.sum(1).double(), Y.sum(1).double()
    def conditional(P, R, sp, sr):
        total = 0.0
        for i in range(0, len(P), 256):
            n11 = (P[i:i + 256] @ R.T).double()
            a, b = sp[i:i + 256, None], sr[None]
            n10, n01 = a - n11, b - n11
            n00 = n - n11 - n10 - n01
            h11, h00, h10, h01 = _h(n11, n), _h(n00, n), _h(n10, n), _h(n01, n)
            same = (torch.minimum(n11, n00) == torch.minimum(n01, n10)) & (torch.maximum(n11, n00) == torch.maximum(n01, n10))
            cand = h11 + h00 + h10 + h01 - (_h(b, n) + _h(n - b, n))
            cand = torch.where((h11 + h00 > h01 + h10) & ~same, cand, float("inf")).min(1).values
            H = _h(a[:, 0], n) + _h(n - a[:, 0], n)
            t = torch.minimum(cand, H).clamp(min=0.0)
            total += float(torch.where(H > 0, t / H.clamp(min=1e-300), torch.zeros_like(H)).sum())
        return total / len(P)
    return 1.0 - 0.5 * (conditional(X, Y, sx, sy) + conditional(Y, X, sy, sx))


def exact(case, seed):
    if case["kind"] == "nmi":
        st = prepare(case, seed)
        n, dense = case["n"], []
        for ptr, nodes in (st["a"], st["b"]):
            m = torch.zeros(len(ptr) - 1, n, device=DEV)
            m[torch.repeat_interleave(torch.arange(len(ptr) - 1), torch.from_numpy(np.diff(ptr))).to(DEV),
              torch.from_numpy(nodes).to(DEV).long()] = 1.0
            dense.append(m)
        return _nmi_dense(dense[0], dense[1], n)
    if case["kind"] != "run" or case["graph"] != "planted":
        return None  # a plain growth of these takes far longer
    n = case["n"]
    rp, col, w, _ = _graph("planted", n, case["deg"], case["weighted"], _gen(seed))
    A = torch.zeros(n, n, dtype=torch.float64, device=DEV)
    src = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
    A[src, col.long()] = 1.0 if w is None else w.double()
    S = case["scales"]
    fit, covers = [], []
    for s in range(S):  # the scales of Sec. 4, finest first
        alpha = case["hi"] if S == 1 else case["lo"] + (case["hi"] - case["lo"]) * (1 - math.log(s + 1) / math.log(S))
        M, f = _grow_dense(A, A.sum(1), alpha)
        first = {}
        for u in range(n):
            first.setdefault(M[u].tobytes(), u)
        rep = sorted(first.values())
        fit.append(f[rep])
        covers.append(torch.from_numpy(M[rep]).to(DEV).float())
    nmi = np.array([_nmi_dense(covers[s], covers[s + 1], n) for s in range(S - 1)])
    win = {}
    for p in (3, 5):
        out = np.full(S, np.nan)
        for i in range(S):
            lo = i - (p - 1) // 2
            w_ = nmi[max(lo, 0):max(min(lo + p - 1, S - 1), 0)]
            if len(w_):
                out[i] = w_.mean()
        win["win%d" % p] = out
    room = np.zeros(S * n)
    for s, f in enumerate(fit):
        room[s * n:s * n + len(f)] = f
    return dict(fitness=room, stability=(nmi, win["win3"], win["win5"]))
