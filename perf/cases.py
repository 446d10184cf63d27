"""The calls whose time matters to a user of this library, as measurable cases.

listed() names them, draw() gives more of the same ranges, prepare() makes
what a program holds before the call (a graph, a partition, a context or a
server), run() is one call through the public entry points, and exact() gives
what can be computed directly.  Graphs are drawn on the GPU with the recipes
of the repository's synthetic inputs (Chung-Lu, R-MAT, random geometric), so
that large ones are quick to make; everything follows from the seed.
"""
from __future__ import annotations

import math
from dataclasses import dataclass
from typing import Optional

import numpy as np
import torch

import paper_2308_15494_gb300 as upr

# What a case does with its graph(s).
#   refine   a kept context refines a partition resident on the device
#   oneshot  a context is created for the graph, refines once and is destroyed
#   rebind   a kept context is bound to a graph in page-locked host memory, refines, result on the host
#   batch    one context over many graphs of different k
#   cut      cut and block weights of a partition, with a context or without any allocation
#   served   a burst of jobs through the continuous-batching server
BASE = {"kind": "refine", "graph": "rmat", "n": 1 << 18, "deg": 32.0, "gamma": 2.2, "weights": "unit", "k": 8,
        "eps": 0.03, "rounds": 8, "schedule": 0, "lp_rounds": 0, "graphs": 1, "count": 1}


def _case(name, **over):
    c = dict(BASE)
    c.update(over)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest graph of the batch and serving workloads, alone: latency and launches only.
        _case("refine_small", graph="chung_lu", n=1024, deg=8.0, k=2, rounds=4),
        # The small single-graph workload (power-law graph, eight blocks).
        _case("refine_16k", graph="chung_lu", n=16384, deg=16.0, k=8, rounds=4),
        # The middle job of the served mix, as a single call with every parameter at its default.
        _case("refine_s18", graph="rmat", n=1 << 18, k=8),
        # A coarse level of a multilevel partitioner: node and edge weights, a size and a k that are
        # no powers of two (k = 23 is one of the paper's block counts).
        _case("refine_weighted_odd", graph="chung_lu", n=1000003, deg=16.0, weights="small", k=23),
        # The weighted mesh-like workload with many blocks (hashed gain-table rows).
        _case("refine_rgg_k256", graph="rgg", n=1 << 22, deg=12.0, weights="heavy", k=256),
        # The headline workload, as the benchmark runs it: all rounds of a call as one CUDA graph.
        _case("refine_s22_k64", graph="rmat", n=1 << 22, k=64, graphs=2),
        # The paper's full pipeline: label propagation, then the final configuration's ten rounds.
        _case("refine_paper", graph="rmat", n=1 << 21, k=32, rounds=10, schedule=6, lp_rounds=5),
        # One refinement of a new graph that lives on the device: a level of a multilevel
        # partitioner, whose graph is used once.
        _case("oneshot_s19", kind="oneshot", graph="rmat", n=1 << 19, k=16),
        # A service that refines one graph after another from page-locked host memory.
        _case("rebind_s20", kind="rebind", graph="rmat", n=1 << 20, k=64, graphs=2),
        # Many independent graphs of different k in one context (the batch workload, a quarter of it).
        _case("batch_1024", kind="batch", graph="chung_lu", n=1 << 16, rounds=4, graphs=2, count=1024),
        # Evaluating a partition: exact cut and block weights of the headline graph.
        _case("cut_s22", kind="cut", graph="rmat", n=1 << 22, k=64),
        # A burst of the served mix: half small graphs, two fifths middle ones, a tenth large ones.
        _case("served_40", kind="served", graph="rmat", n=1 << 21, count=40),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["refine", "oneshot", "rebind", "batch", "cut", "served"], [10, 2, 2, 2, 1, 1])[0]
    c = _case(None, kind=kind, eps=rng.choice([0.01, 0.03, 0.03, 0.1]))
    if kind == "batch":
        c.update(graph="chung_lu", n=_log_int(rng, 2048, 65536), count=_log_int(rng, 16, 1000),
                 rounds=rng.randint(2, 6), graphs=rng.choice([1, 2]))
        return c
    if kind == "served":
        c.update(n=_log_int(rng, 1 << 16, 1 << 20), count=_log_int(rng, 10, 40))
        return c
    c["graph"] = rng.choice(["chung_lu", "rmat", "rgg"])
    top = (1 << 22) if kind in ("refine", "cut") else (1 << 20)
    c["n"] = _log_int(rng, 1000, top) if rng.random() < 0.7 else 1 << rng.randint(10, top.bit_length() - 1)
    c["deg"] = rng.uniform(4.0, 32.0) if c["graph"] != "rgg" else rng.uniform(6.0, 16.0)
    c["gamma"] = rng.uniform(2.1, 2.8)
    c["weights"] = rng.choice(["unit", "unit", "small", "heavy"])
    ks = [k for k in (2, 3, 4, 5, 8, 11, 16, 17, 23, 32, 64, 100, 128, 256) if 64 * k <= c["n"]]
    c["k"] = rng.choice(ks)
    c["rounds"] = rng.randint(2, 8)
    if kind == "refine":
        c["schedule"] = rng.choice([0, 0, 0, 6])
        c["lp_rounds"] = rng.choice([0, 0, 0, 5])
    c["graphs"] = rng.choice([1, 1, 2])
    # no drawn case beyond the headline workload's table and adjacency
    while c["n"] * c["k"] * (c["rounds"] + 2 * c["lp_rounds"]) > (1 << 22) * 64 * 8:
        c["n"] //= 2
    return c


# ------------------------------------------------------------------ graphs
def _csr(n, src, dst):
    """Symmetric CSR without self loops and parallel edges (device tensors)."""
    keep = src != dst
    src, dst = src[keep], dst[keep]
    key = torch.unique(torch.cat([(src << 32) | dst, (dst << 32) | src]))
    rows = key >> 32
    adj = (key & 0xFFFFFFFF).to(torch.int32)
    xadj = torch.zeros(n + 1, dtype=torch.int64, device=key.device)
    xadj[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return xadj, adj


def _chung_lu(ns, degs, gammas, gen):
    """The disjoint union of Chung-Lu graphs: endpoints by the inverse of the
    (continuous) weight distribution (i + 1)^(-1 / (gamma - 1)), ids permuted
    within each graph."""
    dev = "cuda"
    ns_t = torch.tensor(ns, dtype=torch.int64, device=dev)
    off = torch.zeros(len(ns) + 1, dtype=torch.int64, device=dev)
    off[1:] = torch.cumsum(ns_t, 0)
    total = int(sum(ns))
    edges = torch.tensor([int(d * n / 2) for d, n in zip(degs, ns)], dtype=torch.int64, device=dev)
    a = torch.tensor([1.0 - 1.0 / (g - 1.0) for g in gammas], dtype=torch.float64, device=dev)
    gid = torch.repeat_interleave(torch.arange(len(ns), device=dev), edges)
    span = torch.pow(ns_t.double() + 1.0, a) - 1.0

    def endpoint():
        u = torch.rand(len(gid), dtype=torch.float64, device=dev, generator=gen)
        x = torch.pow(1.0 + u * span[gid], (1.0 / a)[gid]) - 1.0
        return torch.minimum(x.long().clamp_(min=0), ns_t[gid] - 1) + off[gid]

    src, dst = endpoint(), endpoint()
    node_gid = torch.repeat_interleave(torch.arange(len(ns), device=dev), ns_t)
    perm = torch.argsort(node_gid.double() + torch.rand(total, dtype=torch.float64, device=dev, generator=gen),
                         stable=True)
    xadj, adj = _csr(total, perm[src], perm[dst])
    return xadj, adj, off, node_gid


def _rmat(n, deg, gen):
    """R-MAT (0.57, 0.19, 0.19) on the next power of two, ids permuted; for
    other n the nodes with the largest new ids are left out."""
    scale = max(1, (n - 1).bit_length())
    full = 1 << scale
    ne = int(deg / 2 * n * (full / n) ** 2)
    src = torch.zeros(ne, dtype=torch.int64, device="cuda")
    dst = torch.zeros(ne, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        x = torch.rand(ne, device="cuda", generator=gen)
        src = (src << 1) | (x >= 0.76)
        dst = (dst << 1) | (((x >= 0.57) & (x < 0.76)) | (x >= 0.95))
    perm = torch.randperm(full, device="cuda", generator=gen)
    src, dst = perm[src], perm[dst]
    if full != n:
        keep = (src < n) & (dst < n)
        src, dst = src[keep], dst[keep]
    return _csr(n, src, dst)


def _rgg(n, deg, gen):
    """Random geometric graph in the unit square, ids in grid-cell order;
    returns the x coordinates as well."""
    dev = "cuda"
    radius = math.sqrt(deg / (math.pi * n))
    g = max(1, int(1.0 / radius))
    xy = torch.rand(n, 2, dtype=torch.float64, device=dev, generator=gen)
    cell = (xy * g).long().clamp_(max=g - 1)
    order = torch.argsort(cell[:, 0] * g + cell[:, 1], stable=True)
    xy, cell = xy[order], cell[order]
    cx, cy = cell[:, 0], cell[:, 1]
    start = torch.zeros(g * g + 1, dtype=torch.int64, device=dev)
    start[1:] = torch.cumsum(torch.bincount(cx * g + cy, minlength=g * g), 0)
    ids = torch.arange(n, device=dev)
    srcs, dsts = [], []
    for dx, dy in ((0, 0), (0, 1), (1, -1), (1, 0), (1, 1)):
        nx, ny = cx + dx, cy + dy
        ok = (nx < g) & (ny >= 0) & (ny < g)
        c1 = (nx * g + ny).clamp(0, g * g - 1)
        lo = torch.where(ok, ids + 1 if (dx, dy) == (0, 0) else start[c1], 0)
        cnt = torch.where(ok, start[c1 + 1], 0) - lo
        src = torch.repeat_interleave(ids, cnt)
        first = torch.cumsum(cnt, 0) - cnt
        dst = lo[src] + torch.arange(len(src), device=dev) - first[src]
        near = ((xy[src] - xy[dst]) ** 2).sum(1) < radius * radius
        srcs.append(src[near])
        dsts.append(dst[near])
    xadj, adj = _csr(n, torch.cat(srcs), torch.cat(dsts))
    return xadj, adj, xy[:, 0]


def _edge_weights(xadj, adj, hi, salt):
    """Symmetric weights in [1, hi] from a hash of the endpoint pair."""
    n = len(xadj) - 1
    u = torch.repeat_interleave(torch.arange(n, device=adj.device), xadj[1:] - xadj[:-1])
    v = adj.long()
    h = torch.minimum(u, v) * 0x9E3779B97F4A7 + torch.maximum(u, v) * 0x2545F4914F6CD + salt * 7919
    h = (h ^ ((h >> 29) & 0x7FFFFFFFF)) * 0x1B873593CC9E2D51
    return (1 + ((h >> 33) & 0x3FFFFFFF) % hi).to(torch.int32)


def _node_weights(n, law, gen):
    if law == "small":
        return torch.randint(1, 9, (n,), dtype=torch.int32, device="cuda", generator=gen)
    cdf = torch.cumsum(torch.arange(1, 1025, dtype=torch.float64, device="cuda") ** -1.5, 0)
    u = torch.rand(n, dtype=torch.float64, device="cuda", generator=gen) * cdf[-1]
    return (1 + torch.searchsorted(cdf, u, right=True).clamp_(max=1023)).to(torch.int32)


def _balanced(n, k, vwgt, gen):
    """Random balanced partition; with weights the heaviest nodes are dealt first, back and forth."""
    perm = torch.randperm(n, device="cuda", generator=gen)
    rank = torch.arange(n, device="cuda")
    if vwgt is not None:
        perm = perm[torch.argsort(vwgt[perm], descending=True, stable=True)]
        pos = rank % (2 * k)
        block = torch.where(pos < k, pos, 2 * k - 1 - pos)
    else:
        block = rank % k
    part = torch.empty(n, dtype=torch.int32, device="cuda")
    part[perm] = block.to(torch.int32)
    return part


def _strips(x, k, vwgt):
    """Vertical strips of equal weight."""
    order = torch.argsort(x, stable=True)
    w = torch.ones(len(x), dtype=torch.int64, device=x.device) if vwgt is None else vwgt.long()
    total = int(w.sum())
    before = torch.cumsum(w[order], 0) - w[order]
    part = torch.empty(len(x), dtype=torch.int32, device=x.device)
    part[order] = (before * k // total).clamp_(max=k - 1).to(torch.int32)
    return part


def _eps(part, vwgt, k, eps):
    """The smallest eps of a 0.01 grid, at least the given one, that admits the partition."""
    w = None if vwgt is None else vwgt.double()
    load = int(torch.bincount(part, weights=w, minlength=k).max())
    total = len(part) if vwgt is None else int(vwgt.long().sum())
    while load > (-(-total // k)) * (1000000 + round(eps * 1e6)) // 1000000:
        eps = round(eps + 0.01, 2)
    return eps


def _single(case, gen):
    """(xadj, adj, vwgt, adjw, part, eps) of a one-graph case, on the device."""
    n, k, x = case["n"], case["k"], None
    if case["graph"] == "chung_lu":
        xadj, adj, _, _ = _chung_lu([n], [case["deg"]], [case["gamma"]], gen)
    elif case["graph"] == "rmat":
        xadj, adj = _rmat(n, case["deg"], gen)
    else:
        xadj, adj, x = _rgg(n, case["deg"], gen)
    vwgt = adjw = None
    if case["weights"] != "unit":
        vwgt = _node_weights(n, case["weights"], gen)
        adjw = _edge_weights(xadj, adj, 9 if case["weights"] == "small" else 64, n)
    part = _strips(x, k, vwgt) if x is not None else _balanced(n, k, vwgt, gen)
    return xadj, adj, vwgt, adjw, part, _eps(part, vwgt, k, case["eps"])


def _many(case, count, gen, rng):
    """count Chung-Lu graphs of the batch workload: n log-uniform from 2^10 to
    the case's n, average degree U[4, 32], exponent U[2.05, 2.8], k from
    {2, 4, 8, 16, 32}, random balanced partitions.  rng draws the sizes, gen the graphs."""
    top = math.log2(case["n"])
    ns = [int(round(2.0 ** rng.uniform(10.0, top))) for _ in range(count)]
    ks = [int(rng.choice([2, 4, 8, 16, 32])) for _ in range(count)]
    degs = [float(rng.uniform(4.0, 32.0)) for _ in range(count)]
    gammas = [float(rng.uniform(2.05, 2.8)) for _ in range(count)]
    xadj, adj, off, gid = _chung_lu(ns, degs, gammas, gen)
    order = torch.argsort(gid.double() + torch.rand(len(gid), dtype=torch.float64, device="cuda", generator=gen),
                          stable=True)
    part = torch.empty(len(gid), dtype=torch.int32, device="cuda")
    rank = torch.arange(len(gid), device="cuda") - off[gid]
    part[order] = (rank % torch.tensor(ks, device="cuda")[gid]).to(torch.int32)
    adj = adj - torch.repeat_interleave(off[gid], xadj[1:] - xadj[:-1]).to(torch.int32)
    starts = off.tolist()
    ends = xadj[off].tolist()
    graphs = [((xadj[starts[i]:starts[i + 1] + 1] - ends[i]).contiguous(), adj[ends[i]:ends[i + 1]])
              for i in range(count)]
    return graphs, ks, part, starts


# ------------------------------------------------------------------- cases
@dataclass
class _Job:
    """A job as Server.submit takes it (host arrays)."""
    xadj: np.ndarray
    adj: np.ndarray
    vwgt: Optional[np.ndarray]
    adjw: Optional[np.ndarray]
    k: int
    eps: float
    part: np.ndarray
    rounds: int


def _params(case):
    p = upr.upr_params_default()
    p.schedule, p.lp_rounds, p.graphs = case["schedule"], case["lp_rounds"], case["graphs"]
    return p


def _pinned(t):
    return None if t is None else t.cpu().pin_memory()


def _served_jobs(case, gen, rng):
    """Half small Chung-Lu graphs, two fifths R-MAT graphs of an eighth of the
    case's n, a tenth of its n, interleaved; the R-MAT graphs come from pools
    of four and one and are asked for with k of 8 and 64 in turn."""
    count = case["count"]
    small = _many(dict(case, n=1 << 16), count // 2, gen, rng)
    jobs = []
    graphs, ks, part, starts = small
    for i, (xa, ad) in enumerate(graphs):
        jobs.append(_Job(xa.cpu().numpy(), ad.cpu().numpy(), None, None, ks[i], case["eps"],
                         part[starts[i]:starts[i + 1]].cpu().numpy(), 4))

    def pool(n, size, total):
        made = []
        for _ in range(size):
            xa, ad = _rmat(n, 32.0, gen)
            parts = {k: _balanced(n, k, None, gen).cpu().numpy() for k in (8, 64)}
            made.append((xa.cpu().numpy(), ad.cpu().numpy(), parts))
        for i in range(total):
            xa, ad, parts = made[i % size]
            k = 64 if (i // size + i) % 2 else 8
            jobs.append(_Job(xa, ad, None, None, k, case["eps"], parts[k], 8))

    pool(max(1024, case["n"] // 8), 4, count * 2 // 5)
    pool(case["n"], 1, max(1, count // 10))
    return [jobs[i] for i in rng.permutation(len(jobs))]


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rng = np.random.Generator(np.random.PCG64([case["n"], case["count"]]))      # sizes: by the case alone
    kind = case["kind"]
    state = {"case": case}
    if kind == "batch":
        graphs, ks, part, _ = _many(case, case["count"], gen, rng)
        graphs = [(xa, ad, None, None) for xa, ad in graphs]
        state["ctx"] = upr.upr_batch_create_mixed(graphs, ks, case["eps"], params=_params(case))
        state["part"] = part
    elif kind == "served":
        state["jobs"] = _served_jobs(case, gen, rng)
        state["server"] = upr.Server()
    else:
        xadj, adj, vwgt, adjw, part, eps = _single(case, gen)
        state.update(eps=eps, part=part)
        if kind in ("oneshot", "cut"):
            state["graph"] = (xadj, adj, vwgt, adjw)
        if kind in ("refine", "cut"):
            state["ctx"] = upr.upr_create(xadj, adj, case["k"], eps, vwgt=vwgt, adjw=adjw, params=_params(case))
        if kind == "rebind":
            host = [_pinned(t) for t in (xadj, adj, vwgt, adjw)]
            state["pinned"] = host
            state["graph"] = [None if t is None else t.numpy() for t in host]
            state["part"] = _pinned(part)
            state["out"] = torch.empty_like(state["part"]).pin_memory()
            xa, ad, vw, aw = state["graph"]
            state["ctx"] = upr.upr_create(xa, ad, case["k"], eps, vwgt=vw, adjw=aw, params=_params(case))
    torch.cuda.synchronize()
    return state


def run(state):
    case = state["case"]
    kind, rounds = case["kind"], case["rounds"]
    if kind == "refine":
        part = state["part"].clone()
        st = upr.upr_refine(state["ctx"], part, rounds)
        return [part, st.cut_in, st.cut_out]
    if kind == "oneshot":
        xadj, adj, vwgt, adjw = state["graph"]
        ctx = upr.upr_create(xadj, adj, case["k"], state["eps"], vwgt=vwgt, adjw=adjw, params=_params(case))
        part = state["part"].clone()
        st = upr.upr_refine(ctx, part, rounds)
        upr.upr_destroy(ctx)
        return [part, st.cut_in, st.cut_out]
    if kind == "rebind":
        xadj, adj, vwgt, adjw = state["graph"]
        upr.upr_rebind(state["ctx"], xadj, adj, case["k"], state["eps"], vwgt=vwgt, adjw=adjw)
        state["out"].copy_(state["part"])
        st = upr.upr_refine(state["ctx"], state["out"].numpy(), rounds)
        return [state["out"], st.cut_in, st.cut_out]
    if kind == "batch":
        part = state["part"].clone()
        status, cut_in, cut_out, _ = upr.upr_batch_refine(state["ctx"], part, rounds)
        return [part, cut_in, cut_out, status]
    if kind == "cut":
        xadj, adj, vwgt, adjw = state["graph"]
        cut, bw = upr.upr_cut(state["ctx"], state["part"])
        cut_n, bw_n = upr.upr_cut_noalloc(xadj, adj, state["part"], case["k"], vwgt=vwgt, adjw=adjw)
        return [cut, bw, cut_n, bw_n]
    server = state["server"]
    tickets = [server.submit(job) for job in state["jobs"]]
    done = [server.wait(t) for t in tickets]
    return [part for part, _, _ in done] + [np.array([cut for _, cut, _ in done], np.int64)]


def work(case):
    """Bytes: the graph and the partition read once, the refined partition
    (or the block weights) written once.  Operations: one addition per
    adjacency entry (the gain table, or the cut).  Edges that the generators
    draw twice are counted once per draw."""
    def one(n, m, weights, out):
        b = 8 * (n + 1) + 4 * m + 4 * n + out
        return b + (0 if weights == "unit" else 4 * m + 4 * n), m

    kind, n = case["kind"], case["n"]
    if kind == "batch":
        lo, hi = 1024.0, float(n)
        mean = (hi - lo) / math.log(hi / lo) if hi > lo else lo
        b, m = one(mean, 18.0 * mean, "unit", 4 * mean)
        return {"bytes": int(b * case["count"]), "flops": int(m * case["count"])}
    if kind == "served":
        cnt = case["count"]
        mean = (65536.0 - 1024.0) / math.log(64.0)
        parts = [(cnt // 2, mean, 18.0 * mean), (cnt * 2 // 5, n / 8, 32.0 * n / 8), (max(1, cnt // 10), n, 32.0 * n)]
        both = [(c * b, c * m) for c, nn, mm in parts for b, m in [one(nn, mm, "unit", 4 * nn)]]
        return {"bytes": int(sum(b for b, _ in both)), "flops": int(sum(m for _, m in both))}
    m = case["deg"] * n
    out = 8 * case["k"] if kind == "cut" else 4 * n
    b, ops = one(n, m, case["weights"], out)
    if kind == "cut":               # both entry points read it all
        b, ops = 2 * b, 2 * ops
    return {"bytes": int(b), "flops": int(ops)}


def _cut_of(xadj, adj, adjw, part):
    n = len(xadj) - 1
    rows = torch.repeat_interleave(torch.arange(n, device=adj.device), xadj[1:] - xadj[:-1])
    cut = part[rows] != part[adj.long()]
    return int((cut if adjw is None else adjw.long()[cut]).sum()) // 2


def exact(case, seed):
    """The cut of the input and, for cut cases, the block weights; a refined
    partition has no value other than the library's own."""
    if case["kind"] in ("batch", "served"):
        return None
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    xadj, adj, vwgt, adjw, part, _ = _single(case, gen)
    cut = _cut_of(xadj, adj, adjw, part)
    if case["kind"] != "cut":
        return [None, cut, None]
    w = torch.ones(case["n"], dtype=torch.float64, device="cuda") if vwgt is None else vwgt.double()
    bw = torch.bincount(part, weights=w, minlength=case["k"]).long().cpu().numpy()
    return [cut, bw, cut, bw]
