"""Graphs on both sides of the rules that leave the core rounds for the
level-wise peel (integer results: tolerance 0)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2001_06784_gb300 import graphgen
from tests.test_gpu_parity import gpu_dag
from tests.test_gpu_paths import band, disjoint, mesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pvt():
    import paper_2001_06784_gb300 as p
    return p


def grid3(a):
    i = np.arange(a ** 3).reshape(a, a, a)
    return graphgen.from_edges(a ** 3, np.concatenate([np.stack([i[1:].ravel(), i[:-1].ravel()], 1),
                                                       np.stack([i[:, 1:].ravel(), i[:, :-1].ravel()], 1),
                                                       np.stack([i[:, :, 1:].ravel(), i[:, :, :-1].ravel()], 1)]))


GRAPHS = {
    # random graphs of low cores around the sizes from which round 20 is looked at,
    # and up to which a low core is enough to leave the rounds there
    "sparse 40k": lambda: graphgen.generate(40_000, er_avg_deg=9.0, seed=1),
    "sparse 300k": lambda: graphgen.generate(300_000, er_avg_deg=5.2, seed=2),
    "less sparse 300k": lambda: graphgen.generate(300_000, er_avg_deg=9.9, seed=3),
    "sparse 32k": lambda: graphgen.generate(32_767, er_avg_deg=5.2, seed=4),
    # many vertices at rounds 20 and 32: bands of three sizes; a lattice
    "band 40k": lambda: band(40_000, 9),
    "band 6k": lambda: band(6_000, 12),
    "band 2k": lambda: band(2_000, 20),
    "bands and a clique": lambda: disjoint(*[band(400, 8) for _ in range(100)], band(40, 39)),
    "lattice": lambda: grid3(33),
    # a dense core, and chains beside it that end late
    "core and a mesh": lambda: disjoint(graphgen.generate(20_000, chung_lu=(200_000, 2.1), seed=5), mesh(130, 130)),
    "core and a band": lambda: disjoint(graphgen.generate(20_000, chung_lu=(200_000, 2.1), seed=6), band(900, 3)),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_core_rules(pvt, name):
    """Core numbers equal the oracle's, out-degrees stay within them, every edge
    is in one out-list, and the orientation has no cycle (every strongly
    connected component is one vertex)."""
    from scipy.sparse import csr_matrix
    from scipy.sparse.csgraph import connected_components
    rp, col = GRAPHS[name]()
    n = len(rp) - 1
    _, core, _ = oracle.orient(rp, col)
    dag = gpu_dag(pvt, rp, col)
    assert np.array_equal(dag.cores().cpu().numpy().view(np.uint32), core)
    assert dag.alpha == int(core.max())
    orow, ocol = (t.cpu().numpy() for t in dag.out_lists())
    outdeg = np.diff(orow)
    assert (outdeg <= core.astype(np.int64)).all()
    dag_m = csr_matrix((np.ones(len(ocol), np.int8), ocol, orow), shape=(n, n))
    both = dag_m + dag_m.T
    both.sort_indices()
    assert np.array_equal(both.indptr, rp) and np.array_equal(both.indices, col.astype(np.int64)) and both.max() == 1
    assert connected_components(dag_m, directed=True, connection="strong", return_labels=False) == n
    dag.free()
