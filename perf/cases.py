"""What the clique-count library is timed on: its work as a program has it do,
through the public entry points, from a query of a few hundred vertices to the
1M-vertex all-k count of the benchmark.

A case is a dict of plain values.  Its "kind" says which call it stands for:

  query   a program with a CSR on the GPU asks for all counts of a graph it has
          not seen: orient, core numbers, global counts, release
  cores   the degeneracy orientation and the core numbers alone (the k-core
          decomposition), as a pre-pass over a larger graph
  global  counts of every k on a graph that is already oriented, as a program
          does that keeps the oriented graph and asks again (other k, other W)
  vertex  the per-vertex table c_k(v) of an oriented graph
  edge    the per-edge table c_k(e) of an oriented graph
  serve   a burst of independent queries through the query server, host CSRs in
          and host tables out

Graphs are the repository's synthetic stand-ins for social and web networks:
Chung-Lu power laws (or Erdos-Renyi) with planted dense communities or cliques.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2001_06784_gb300 as pvt

DEVICE = "cuda:0"


def listed():
    return [
        # the smallest query: a few hundred vertices, where launches, copies
        # and synchronisations are the time
        dict(name="query_n300", kind="query", n=300, deg=14.0, beta=0.0, groups=2, smin=24, smax=24, rho=1.0, kmax=0,
             W=0),
        # the repository's small workload: ER of 2,000 vertices, average degree
        # 20, one planted 30-clique, all k
        dict(name="query_er2k", kind="query", n=2000, deg=20.45, beta=0.0, groups=1, smin=30, smax=30, rho=1.0, kmax=0,
             W=0),
        # an ordinary query: a power-law graph of odd size with communities
        dict(name="query_cl61k", kind="query", n=61_013, deg=14.1, beta=2.2, groups=40, smin=15, smax=45, rho=0.9,
             kmax=48, W=1),
        # the benchmark's workload: 1M vertices, 10.8M edges, 500 communities
        dict(name="query_cl1m", kind="query", n=1_000_000, deg=21.6, beta=2.1, groups=500, smin=20, smax=60, rho=0.9,
             kmax=64, W=3),
        # k-core decomposition of a larger, sparser graph
        dict(name="cores_cl2m", kind="cores", n=2_000_003, deg=16.0, beta=2.3, groups=0, smin=0, smax=0, rho=0.0,
             kmax=0, W=0),
        # every k again on an oriented graph of 500k vertices, 8M edges
        dict(name="global_cl500k", kind="global", n=500_000, deg=33.0, beta=2.3, groups=200, smin=15, smax=40, rho=1.0,
             kmax=48, W=2),
        # counts for k <= 4 of a social-shaped graph with a dense core
        # (degeneracy above 256: the widest roots)
        dict(name="global_k4_dense300k", kind="global", n=300_000, deg=80.0, beta=2.0, groups=0, smin=0, smax=0,
             rho=0.0, kmax=4, W=6),
        # per-vertex tables: every k that the planted cliques reach, and k <= 5
        # of a graph of ragged size with communities
        dict(name="vertex_cl500k", kind="vertex", n=500_000, deg=33.0, beta=2.3, groups=200, smin=15, smax=40,
             rho=1.0, kmax=40, W=2),
        dict(name="vertex_k5_cl90k", kind="vertex", n=90_001, deg=25.1, beta=2.2, groups=30, smin=12, smax=40, rho=0.9,
             kmax=5, W=2),
        # per-edge tables: k <= 12 of 2M edges, and every k of one small graph
        dict(name="edge_k12_cl130k", kind="edge", n=130_007, deg=31.6, beta=2.3, groups=60, smin=15, smax=40, rho=1.0,
             kmax=12, W=2),
        dict(name="edge_cl5k", kind="edge", n=5003, deg=22.4, beta=2.3, groups=4, smin=10, smax=22, rho=1.0, kmax=22,
             W=1),
        # the serving stream's shape: independent queries, n log-uniform, global
        # or per-edge, small ones batched and large ones on the whole GPU
        dict(name="serve_48", kind="serve", n=30_011, queries=48, kmax=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) | 1


def draw(rng):
    kind = rng.choice(["query", "query", "query", "cores", "global", "vertex", "edge", "serve"])
    if kind == "serve":
        return dict(kind=kind, n=_log(rng, 1000, 30_000), queries=rng.randint(4, 48), kmax=rng.choice([4, 8, 16]))
    top = {"query": 1_000_000, "cores": 2_000_000, "global": 500_000, "vertex": 300_000, "edge": 130_000}[kind]
    n = _log(rng, 300, top)
    deg = round(rng.uniform(8.0, 21.0 if n > 300_000 else 31.0), 2)
    beta = 0.0 if rng.random() < 0.3 else round(rng.uniform(2.1, 2.5), 3)
    smin = rng.randint(8, 20)
    smax = smin + rng.randint(0, 25)
    groups = 0 if kind == "cores" else rng.randint(0, max(1, min(400, n // 1500)))
    kmax = {"query": 48, "cores": 0, "global": rng.choice([48, 48, 3, 5, 8]), "vertex": rng.randint(3, 30),
            "edge": rng.randint(3, 12)}[kind]
    # words that hold every count: n * 2^alpha for a degeneracy above any that
    # these graphs have
    alpha = max(0.75 * deg + 0.055 * math.sqrt(n * deg), smax + 12)
    W = int(n.bit_length() + alpha + 1 + 63) // 64
    return dict(kind=kind, n=n, deg=deg, beta=beta, groups=groups, smin=smin, smax=smax, rho=rng.choice([0.8, 0.9, 1.0]),
                kmax=kmax, W=W)


# ---------------------------------------------------------------- graphs

def _chung_lu_cdf(n, m, beta):
    """Cumulative vertex weights of the repository's Chung-Lu recipe: weights
    (i + i0)^(-1/(beta-1)), i0 the smallest offset for which the largest
    expected degree stays at most sqrt(2m)."""
    e = -1.0 / (beta - 1.0)
    i = np.arange(n, dtype=np.float64)
    lo, hi = 1.0, float(n)
    for _ in range(40):
        mid = math.sqrt(lo * hi)
        w = (i + mid) ** e
        if 2.0 * m * w[0] / w.sum() <= math.sqrt(2.0 * m):
            hi = mid
        else:
            lo = mid
    return np.cumsum((i + hi) ** e)


def _keys(a, b, n):
    return (torch.minimum(a, b) * n + torch.maximum(a, b))[a != b]


def _graph(case, seed):
    """(row_ptr int64[n+1], col int32[2m]) on the GPU: simple, sorted, symmetric,
    exactly n * deg / 2 edges, the planted groups' among them."""
    n = case["n"]
    m = int(n * case["deg"] / 2)
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    planted = torch.empty(0, dtype=torch.int64, device=DEVICE)
    if case["groups"]:
        # planted groups: uniform distinct members, each pair an edge with
        # probability rho
        size = torch.randint(case["smin"], case["smax"] + 1, (case["groups"], 1), generator=g, device=DEVICE)
        step = torch.randint(1, max(n // case["smax"], 2), (case["groups"], case["smax"]), generator=g, device=DEVICE)
        mem = torch.cumsum(step, 1) % n
        iu = torch.triu_indices(case["smax"], case["smax"], 1, device=DEVICE)
        u, v = mem[:, iu[0]], mem[:, iu[1]]
        keep = iu[1][None, :] < size
        keep &= torch.rand(u.shape, generator=g, device=DEVICE) <= case["rho"]
        planted = torch.unique(_keys(u[keep], v[keep], n))
    cdf = torch.from_numpy(_chung_lu_cdf(n, m, case["beta"])).to(DEVICE) if case["beta"] else None
    want = max(m - planted.numel(), 0)
    rest = torch.empty(0, dtype=torch.int64, device=DEVICE)
    for _ in range(64):
        lack = want - rest.numel()
        if lack <= 0:
            break
        draws = int(lack * 1.1) + 64
        if cdf is None:
            ends = torch.randint(n, (2 * draws,), generator=g, device=DEVICE)
        else:
            r = torch.rand(2 * draws, generator=g, device=DEVICE, dtype=torch.float64) * cdf[-1]
            ends = torch.searchsorted(cdf, r, right=True).clamp_(max=n - 1)
        rest = torch.unique(torch.cat([rest, _keys(ends[:draws], ends[draws:], n)]))
        rest = rest[~torch.isin(rest, planted)] if planted.numel() else rest
    rest = rest[torch.randperm(rest.numel(), generator=g, device=DEVICE)[:want]]
    key = torch.cat([planted, rest])
    a, b = key // n, key % n
    both = torch.sort(torch.cat([a * n + b, b * n + a]))[0]
    deg = torch.bincount(both // n, minlength=n)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEVICE)
    torch.cumsum(deg, 0, out=row_ptr[1:])
    return row_ptr, (both % n).to(torch.int32)


def _burst(case):
    """The graphs of a burst: sizes evenly over the logarithm of 100..n, ER and
    Chung-Lu in turn, per-edge and global questions mixed, in a shuffled order
    (the same for every seed; the graphs themselves are the seed's)."""
    rng = random.Random(case["n"] * 64 + case["queries"])
    out = []
    for i in range(case["queries"]):
        t = (i + rng.random()) / case["queries"]
        er = i % 2 == 0
        out.append((dict(n=int(math.exp(math.log(100) + t * math.log(case["n"] / 100))),
                         deg=rng.uniform(5.0, 55.0 if er else 14.0), beta=0.0 if er else rng.uniform(2.0, 2.5), groups=0),
                    "edge" if rng.random() < 0.5 else "global"))
    rng.shuffle(out)
    return out


# ------------------------------------------------------------------ calls

def prepare(case, seed):
    if case["kind"] == "serve":
        queries = []
        for i, (shape, what) in enumerate(_burst(case)):
            row_ptr, col = _graph(shape, seed * 1009 + i)
            queries.append((row_ptr.cpu().numpy(), col.cpu().numpy().view(np.uint32), what))
        return dict(kind="serve", queries=queries, kmax=case["kmax"], server=pvt.Server(mem_budget=64 << 30))
    row_ptr, col = _graph(case, seed)
    state = dict(kind=case["kind"], row_ptr=row_ptr, col=col, kmax=case["kmax"] or None, W=case["W"] or None)
    if case["kind"] in ("global", "vertex", "edge"):
        state["dag"] = pvt.orient(row_ptr, col)
    return state


def run(state):
    kind = state["kind"]
    if kind == "serve":
        sv = state["server"]
        tickets = [sv.submit(rp, col, what, kmax=state["kmax"]) for rp, col, what in state["queries"]]
        out = []
        for t in tickets:
            sv.wait(t)
            out.append(sv.result(t)[0].view(np.int64))
        return out
    if kind in ("query", "cores"):
        dag = pvt.orient(state["row_ptr"], state["col"])
        core = dag.cores()
        out = [core] if kind == "cores" else [core, dag.count_global(kmax=state["kmax"], W=state["W"])]
        dag.free()
        return out
    dag = state["dag"]
    if kind == "global":
        return [dag.count_global(kmax=state["kmax"], W=state["W"])]
    if kind == "vertex":
        return [dag.count_local_vertex(kmax=state["kmax"], W=state["W"])]
    return [dag.count_local_edge(kmax=state["kmax"], W=state["W"])]


def work(case):
    """The CSR read once and the answer written once; one operation per stored
    edge entry.  What the clique tree itself takes depends on the graph and is
    not in these figures."""
    if case["kind"] == "serve":
        total = dict(bytes=0.0, flops=0.0)
        for shape, what in _burst(case):
            m = int(shape["n"] * shape["deg"] / 2)
            total["bytes"] += 8.0 * shape["n"] + 8.0 * m + (8.0 * m * (case["kmax"] + 1) if what == "edge" else 0.0)
            total["flops"] += 2.0 * m
        return total
    n, m = case["n"], int(case["n"] * case["deg"] / 2)
    row = 8.0 * (case["kmax"] + 1) * case["W"]
    out = {"query": 4.0 * n, "cores": 4.0 * n, "global": row, "vertex": n * row, "edge": m * row}[case["kind"]]
    return dict(bytes=8.0 * (n + 1) + 8.0 * m + out, flops=2.0 * m)


# ------------------------------------------------------------- reference

def _core_numbers(row_ptr, col):
    """Core numbers by removing every vertex of degree <= k until none is
    left, k rising (plain torch, 64-bit)."""
    n = row_ptr.numel() - 1
    deg = row_ptr[1:] - row_ptr[:-1]
    col = col.to(torch.int64)
    left, core = deg.clone(), torch.zeros(n, dtype=torch.int64, device=deg.device)
    alive = torch.ones(n, dtype=torch.bool, device=deg.device)
    k = 0
    while bool(alive.any()):
        k = max(k, int(left[alive].min()))
        gone = torch.nonzero(alive & (left <= k)).flatten()
        while gone.numel():
            core[gone] = k
            alive[gone] = False
            cnt = deg[gone]
            at = torch.repeat_interleave(row_ptr[gone] - (torch.cumsum(cnt, 0) - cnt), cnt)
            nb = col[at + torch.arange(at.numel(), device=deg.device)]
            left.sub_(torch.bincount(nb, minlength=n))
            nb = torch.unique(nb)
            gone = nb[alive[nb] & (left[nb] <= k)]
    return core


def _tree_counts(row_ptr, col, core, kmax):
    """C_k, c_k(v) and c_k(e) as Python integers: the pivoted clique tree with
    neighbourhoods as integer bit sets, one root at a time in an order of
    rising core number (small graphs)."""
    n = len(row_ptr) - 1
    order = _removal_order(row_ptr, col)
    rank = [0] * n
    for i, v in enumerate(order):
        rank[v] = i
    C = [0] * (kmax + 1)
    cv = [[0] * (kmax + 1) for _ in range(n)]
    ce = {}
    for v in range(n):
        for u in col[row_ptr[v]:row_ptr[v + 1]]:
            if v < u:
                ce[(v, u)] = [0] * (kmax + 1)
    nbr = [set(col[row_ptr[v]:row_ptr[v + 1]]) for v in range(n)]

    def leaf(hold, piv):
        h, p = len(hold), len(piv)
        for i in range(p + 1):
            if h + i <= kmax:
                C[h + i] += math.comb(p, i)
        mem = [(x, 0) for x in hold] + [(x, 1) for x in piv]
        for a, (x, px) in enumerate(mem):
            for i in range(p - px + 1):
                if h + px + i <= kmax:
                    cv[x][h + px + i] += math.comb(p - px, i)
            for y, py in mem[:a]:
                row, q = ce[(min(x, y), max(x, y))], px + py
                for i in range(p - q + 1):
                    if h + q + i <= kmax:
                        row[h + q + i] += math.comb(p - q, i)

    def walk(S, hold, piv):
        if len(hold) > kmax:
            return
        if not S:
            leaf(hold, piv)
            return
        best = max(S, key=lambda x: len(nbr[x] & S))
        walk(S & nbr[best], hold, piv + [best])
        rest = set(S)
        for v in sorted(S - nbr[best] - {best}):
            rest.discard(v)
            walk(rest & nbr[v], hold + [v], piv)

    for r in range(n):
        walk({u for u in nbr[r] if rank[u] > rank[r]}, [r], [])
    return C, cv, [ce[e] for e in sorted(ce)]


def _removal_order(row_ptr, col):
    n = len(row_ptr) - 1
    deg = [row_ptr[v + 1] - row_ptr[v] for v in range(n)]
    buckets, gone, order, k = {}, [False] * n, [], 0
    for v in range(n):
        buckets.setdefault(deg[v], []).append(v)
    while len(order) < n:
        while not buckets.get(k):
            k += 1
        v = buckets[k].pop()
        if gone[v] or deg[v] != k:
            continue
        gone[v] = True
        order.append(v)
        for u in col[row_ptr[v]:row_ptr[v + 1]]:
            if not gone[u]:
                deg[u] -= 1
                buckets.setdefault(deg[u], []).append(u)
        k = max(k - 1, 0)
    return order


def _words(values, W):
    a = np.zeros((len(values), W), dtype=np.uint64)
    for i, x in enumerate(values):
        for w in range(W):
            a[i, w] = (x >> (64 * w)) & 0xFFFFFFFFFFFFFFFF
    return torch.from_numpy(a.view(np.int64))


def exact(case, seed):
    if case["kind"] == "serve":
        return None
    small = case["n"] * case["deg"] <= 45_000 and not case["beta"]
    if case["kind"] not in ("query", "cores") and not small:
        return None
    row_ptr, col = _graph(case, seed)
    core = _core_numbers(row_ptr, col)
    if case["kind"] == "cores":
        return [core.to(torch.int32).cpu()]
    counts = None
    if small:
        alpha = int(core.max())
        kmax = case["kmax"] or alpha + 1
        W = case["W"] or max(1, (case["n"].bit_length() + alpha + 1 + 63) // 64)
        C, cv, ce = _tree_counts(row_ptr.tolist(), col.tolist(), core, kmax)
        tables = {"query": lambda: _words(C, W), "global": lambda: _words(C, W),
                  "vertex": lambda: torch.stack([_words(x, W) for x in cv]),
                  "edge": lambda: torch.stack([_words(x, W) for x in ce])}
        counts = tables[case["kind"]]()
    return [core.to(torch.int32).cpu(), counts] if case["kind"] == "query" else [counts]
