"""Device memory across streams and failures: what a call leaves in flight when
it returns, and what a dag's release has to wait for (integer results:
tolerance 0)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2001_06784_gb300 import graphgen
from tests.test_gpu_parity import gpu_dag

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pvt():
    import paper_2001_06784_gb300 as p
    return p


@pytest.mark.parametrize("streams", [1, 2])
def test_free_waits_for_the_copies_of_the_core_numbers(pvt, streams):
    """pvt_dag_cores only enqueues its copy.  A dag freed while such copies wait
    behind other work on their streams is released after them: the free returns
    with every copy made."""
    import torch
    rp, col = graphgen.generate(5000, er_avg_deg=12.0, planted=[(2, 20, 30, 0.9)], seed=51)
    _, core, _ = oracle.orient(rp, col)
    dag = gpu_dag(pvt, rp, col)
    torch.cuda.synchronize()
    ss = [torch.cuda.Stream() for _ in range(streams)]
    outs = []
    for s in ss:
        with torch.cuda.stream(s):
            torch.cuda._sleep(100_000_000)  # some 50 ms of the stream's time
            outs.append(dag.cores())
    assert not ss[0].query()
    dag.free()
    assert all(s.query() for s in ss)
    for out in outs:
        assert np.array_equal(out.cpu().numpy().view(np.uint32), core)
