"""The kernels a size rule picks, at the edges of their ranges, against the CPU
oracle (integer results: tolerance 0).

Each case sits on one side of a rule: the gather of the <= 32 class (from 8,192
such roots on), the row widths between powers of two, the table window, parts
and relabelled labels of the local counts, the one-block and grid forms of the
core rounds, and the graphs that leave them for the level-wise peel."""
from __future__ import annotations

import math

import numpy as np
import pytest

import oracle
from paper_2001_06784_gb300 import graphgen
from tests import graphs
from tests.test_gpu_parity import gpu_dag, limbs_as_words

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pvt():
    import paper_2001_06784_gb300 as p
    return p


def disjoint(*parts):
    """Disjoint union of CSR graphs."""
    edges, base = [], 0
    for rp, col in parts:
        edges.append(graphgen.edge_list(rp, col) + base)
        base += len(rp) - 1
    return graphgen.from_edges(base, np.concatenate(edges))


def band(n, w):
    """Vertex i adjacent to i+1 .. i+w: core numbers fall one chain at a time."""
    return graphgen.from_edges(n, np.concatenate([np.stack([np.arange(n - k), np.arange(k, n)], 1) for k in range(1, w + 1)]))


def mesh(a, b):
    i = np.arange(a * b).reshape(a, b)
    return graphgen.from_edges(a * b, np.concatenate([np.stack([i[:, :-1].ravel(), i[:, 1:].ravel()], 1),
                                                      np.stack([i[:-1].ravel(), i[1:].ravel()], 1)]))


def star(leaves):
    return graphgen.from_edges(leaves + 1, np.stack([np.zeros(leaves, np.int64), np.arange(1, leaves + 1)], 1))


# ---------------------------------------------- the gather of the <= 32 class

GATHER = {
    # out-degrees 1, 2 (a pair, adjacent or not), 31, 32 and, beside the class, 33
    "cliques 2 3 32 33 34": lambda: disjoint(graphgen.generate(9000, er_avg_deg=7.0, seed=3),
                                             graphs.disjoint_cliques([2, 3, 32, 33, 34])),
    "below the rule": lambda: graphgen.generate(8000, er_avg_deg=7.0, planted=[(3, 20, 33, 0.9)], seed=4),
    "dense communities": lambda: graphgen.generate(12001, er_avg_deg=9.0, planted=[(6, 24, 40, 0.85)], seed=5),
    "trees and isolated": lambda: disjoint(band(9000, 1), star(300),
                                           graphgen.from_edges(50, np.zeros((0, 2), np.int64))),
}


@pytest.mark.parametrize("name", sorted(GATHER))
@pytest.mark.parametrize("kmax", [1, 2, 3, None])
def test_gather_of_light_roots(pvt, name, kmax):
    rp, col = GATHER[name]()
    ref = oracle.count(rp, col, kmax=-1 if kmax is None else kmax)
    dag = gpu_dag(pvt, rp, col)
    walked = set()
    for chunk, frames, lanes in [(4, True, True), (1, True, True), (32, True, True), (4, False, True), (4, True, False)]:
        dag.set_policy(chunk=chunk, frames=frames, lanes=lanes)
        assert pvt.to_ints(dag.count_global(kmax=ref["kmax"])) == ref["C"], (chunk, frames, lanes)
        st = dag.stats()
        walked.add((st["sct_nodes"], st["sct_leaves"], st["pivot_words"], st["class_words"][1]))
        assert sum(st["class_words"]) + st["frame_words"] == st["pivot_words"]
    assert len(walked) == 1  # the same tree, and the class's share of it, whichever kernels walk it
    hist = dag.count_hist(0, dag.n, kmax=ref["kmax"])
    assert pvt.to_ints(dag.combine_hist(hist, kmax=ref["kmax"])) == ref["C"]
    dag.free()


# ------------------------------------------------- row widths of wide roots

@pytest.mark.parametrize("alpha", [96, 97, 129, 160, 161, 192, 193, 256, 257, 320, 321, 384, 385, 640, 641])
def test_row_widths(pvt, alpha):
    """Largest out-degrees on both sides of every row width, walked by warps and
    by blocks.  K_n less the edges {0,1}, {2,3}, {4,5}: a k-clique takes each
    pair's vertices apart, so C_k = sum_i C(3, i) 2^i C(n - 6, k - i)."""
    n = alpha + 2
    iu = np.stack(np.triu_indices(n, 1), 1)
    rp, col = graphgen.from_edges(n, iu[~((iu[:, 0] < 6) & (iu[:, 0] % 2 == 0) & (iu[:, 1] == iu[:, 0] + 1))])
    want = [0] + [sum(math.comb(3, i) * 2 ** i * math.comb(n - 6, k - i) for i in range(min(3, k) + 1))
                  for k in range(1, 10)]
    dag = gpu_dag(pvt, rp, col)
    assert dag.alpha == alpha
    for cta in ((0,) * 7, (0, 0, 0, 0, 1, 1, 1)):
        dag.set_policy(cta=cta)
        assert pvt.to_ints(dag.count_global(kmax=9)) == want
    dag.free()


def test_recorded_count_after_a_wider_one(pvt):
    """A recorded global count whose table another call has since rebuilt with
    wider entries is recorded anew, not replayed."""
    import torch
    rp, col = graphgen.generate(9000, er_avg_deg=8.0, planted=[(3, 40, 60, 0.8)], seed=9)
    ref = oracle.count(rp, col)
    dag = gpu_dag(pvt, rp, col)
    dag.set_policy(graph=True)
    out = torch.empty((ref["kmax"] + 1, dag.min_words), dtype=torch.int64, device="cuda")
    for W in (0, 0, 1, 0, 0, 2, 0):  # 0: the recorded call
        if W:
            dag.count_local_vertex(kmax=ref["kmax"], W=dag.min_words + W)
        else:
            assert pvt.to_ints(dag.count_global(kmax=ref["kmax"], out=out.zero_())) == ref["C"]
    dag.free()


# ------------------------------------------------------------ local counts

LOCAL = {
    # (graph, sizes): windows of 8, 10 and 12 sizes on both sides, roots in
    # parts, near-cliques, labels of 32 and 33 members below wider roots
    "one word": (lambda: graphgen.generate(700, er_avg_deg=8.0, planted=[(4, 18, 33, 0.9), (2, 14, 14, 1.0)], seed=21),
                 (1, 3, 11, 12, 13, None)),
    "two words": (lambda: graphgen.generate(500, er_avg_deg=9.0, planted=[(3, 36, 60, 0.75)], seed=22), (2, 10, 11)),
    "three words": (lambda: graphs.gnp(150, 0.5, 23), (5, 8, 9)),
    "four words": (lambda: graphs.clique_minus_random(125, 11, 24), (4, 8, 9)),
    "near-cliques": (lambda: disjoint(graphs.clique_minus_random(34, 8, 1), graphs.clique_minus_random(60, 9, 2),
                                      graphs.clique_minus_random(120, 7, 3)), (6, 14)),
}


@pytest.mark.parametrize("name,kmax", [(n, k) for n in sorted(LOCAL) for k in LOCAL[n][1]])
def test_local_tables_at_the_window(pvt, name, kmax):
    rp, col = LOCAL[name][0]()
    ref = oracle.count(rp, col, vertex=True, edge=True, kmax=-1 if kmax is None else kmax)
    dag = gpu_dag(pvt, rp, col)
    W = dag.min_words
    for policy in (dict(), dict(persistent=False)):  # roots in parts, and each by its own warp
        dag.set_policy(**policy)
        cv = dag.count_local_vertex(kmax=ref["kmax"]).cpu().numpy().view(np.uint64)
        assert np.array_equal(cv, limbs_as_words(ref["cv"], W))
        ce = dag.count_local_edge(kmax=ref["kmax"]).cpu().numpy().view(np.uint64)
        assert np.array_equal(ce, limbs_as_words(ref["ce"], W))
        st = dag.stats()
        if kmax is None:  # the tree of the global count
            dag.count_global(kmax=ref["kmax"])
            g = dag.stats()
            assert (st["sct_nodes"], st["sct_leaves"], st["pivot_words"]) == (g["sct_nodes"], g["sct_leaves"], g["pivot_words"])
    dag.free()


def test_local_counts_past_one_word(pvt):
    """K_80: per-edge counts C(78, k-2) pass 2^64, so the low words wrap."""
    rp, col = graphs.complete(80)
    dag = gpu_dag(pvt, rp, col)
    ce = pvt.to_ints(dag.count_local_edge()[:3])
    cv = pvt.to_ints(dag.count_local_vertex()[-2:])
    assert math.comb(78, 39) > 1 << 64
    assert ce == [[0, 0] + [math.comb(78, k - 2) for k in range(2, 81)]] * 3
    assert cv == [[0] + [math.comb(79, k - 1) for k in range(1, 81)]] * 2
    dag.free()


# ------------------------------------------------------------- orientation

ORIENT = {
    "one block": lambda: graphgen.generate(1024, er_avg_deg=15.0, seed=31),
    "one vertex more": lambda: graphgen.generate(1025, er_avg_deg=15.0, seed=31),
    "more entries": lambda: graphgen.generate(1000, er_avg_deg=18.0, planted=[(1, 40, 40, 1.0)], seed=32),
    "rows 32 33 256 257": lambda: disjoint(star(32), star(33), star(256), star(257), graphs.complete(33),
                                           graphs.complete(34), graphs.complete(257), graphs.complete(258)),
    "rows above the clamp": lambda: disjoint(star(5000), graphgen.generate(3000, chung_lu=(40000, 2.0), seed=33)),
    "power law": lambda: graphgen.generate(20011, chung_lu=(200000, 2.1), planted=[(10, 20, 60, 0.8)], seed=34),
    "mesh": lambda: mesh(90, 110),
    "path": lambda: band(3000, 1),
    "thick path": lambda: band(6000, 12),
    "no edges": lambda: graphgen.from_edges(2000, np.zeros((0, 2), np.int64)),
}


@pytest.mark.parametrize("name", sorted(ORIENT))
def test_core_rounds(pvt, name):
    """Core numbers equal the oracle's; the orientation is acyclic by its key
    and every out-degree is at most the vertex's core number."""
    rp, col = ORIENT[name]()
    _, core, _ = oracle.orient(rp, col)
    dag = gpu_dag(pvt, rp, col)
    assert np.array_equal(dag.cores().cpu().numpy().view(np.uint32), core)
    assert dag.alpha == int(core.max())
    orow, ocol = (t.cpu().numpy() for t in dag.out_lists())
    outdeg = np.diff(orow)
    assert outdeg.sum() == len(col) // 2 and (outdeg <= core.astype(np.int64)).all()
    src = np.repeat(np.arange(len(outdeg)), outdeg)
    both = np.concatenate([np.stack([src, ocol], 1), np.stack([ocol, src], 1)])
    want = np.stack([np.repeat(np.arange(len(rp) - 1), np.diff(rp)), col.astype(np.int64)], 1)
    assert np.array_equal(both[np.lexsort((both[:, 1], both[:, 0]))], want)  # each edge once
    ref = oracle.count(rp, col, kmax=4)
    assert pvt.to_ints(dag.count_global(kmax=4)) == ref["C"]
    dag.free()


# ------------------------------------------------------------------ server

def test_server_large_result(pvt):
    """A per-edge table of several copy pieces equals the single-graph call."""
    rp, col = graphgen.generate(6000, er_avg_deg=20.0, planted=[(2, 10, 20, 1.0)], seed=41)
    with pvt.Server(mem_budget=8 << 30) as sv:
        t = sv.submit(rp, col, "edge", kmax=20)
        assert sv.wait(t, 60000)
        got = sv.result(t)[0]
    dag = gpu_dag(pvt, rp, col)
    want = dag.count_local_edge(kmax=20).cpu().numpy().view(np.uint64)
    assert got.nbytes > 4 << 20 and np.array_equal(got, want)
    dag.free()
