"""Labels walked in place by warps: the leaf histogram of a block past the point
at which a warp empties it, in every form (integer results: tolerance 0)."""
from __future__ import annotations

import pytest

from tests import graphs
from tests.test_gpu_parity import gpu_dag

pytestmark = pytest.mark.gpu

DRAIN = 1 << 16  # leaves of a warp (HIST_DRAIN)


def test_walks_past_a_drain():
    """G(100, 0.8), k <= 7: the lane walk's counts and tree, then the forms in
    which one warp walks whole roots."""
    import torch
    import paper_2001_06784_gb300 as pvt
    from paper_2001_06784_gb300 import _lib
    rp, col = graphs.gnp(100, 0.8, 81)
    dag = gpu_dag(pvt, rp, col)
    want = dag.count_global(kmax=7)
    st = dag.stats()
    tree = (st["sct_nodes"], st["sct_leaves"], st["pivot_words"])
    assert st["sct_leaves"] > DRAIN * sum(st["roots"][2:])
    assert pvt.to_ints(want)[1:3] == [100, len(col) // 2]
    for policy in (dict(persistent=False), dict(frames=False), dict(frames=False, split=[0] * 7), dict(lanes=False)):
        dag.set_policy(**policy)
        assert torch.equal(dag.count_global(kmax=7), want), policy
        st = dag.stats()
        assert (st["sct_nodes"], st["sct_leaves"], st["pivot_words"]) == tree, policy
    orow, ocol = dag.out_lists()
    out = torch.zeros_like(want)
    _lib.check(_lib.lib().pvt_count_global_noalloc(dag.n, orow.data_ptr(), ocol.data_ptr(), dag.alpha, 7, dag.min_words,
                                                   out.data_ptr(), torch.cuda.current_stream().cuda_stream))
    assert torch.equal(out, want)
    dag.free()
