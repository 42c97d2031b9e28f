"""Device memory across streams and failures: what a call leaves in flight when
it returns, and what a dag's release has to wait for (integer results:
tolerance 0)."""
from __future__ import annotations

import contextlib
import ctypes

import numpy as np
import pytest

import oracle
from paper_2001_06784_gb300 import graphgen
from tests import graphs
from tests.test_gpu_parity import gpu_dag
from tests.test_gpu_paths import disjoint, mesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pvt():
    import paper_2001_06784_gb300 as p
    return p


class PoolProps(ctypes.Structure):
    """CUmemPoolProps: pinned memory of one device, at most maxSize bytes."""
    _fields_ = [("allocType", ctypes.c_int), ("handleTypes", ctypes.c_int), ("locationType", ctypes.c_int),
                ("locationId", ctypes.c_int), ("security", ctypes.c_void_p), ("maxSize", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


RESERVED_MEM_CURRENT, RESERVED_MEM_HIGH, USED_MEM_CURRENT = 5, 6, 7  # CU_MEMPOOL_ATTR_*


@contextlib.contextmanager
def limited_pool(limit):
    """Stream-ordered allocations come from a pool of at most `limit` bytes:
    beyond it they fail as on a full device.  Yields a function that gives one
    of its figures (the bytes in use).  The pool itself stays: what was allocated from it may live
    on."""
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    torch.cuda.synchronize()
    pool, usual = ctypes.c_void_p(), ctypes.c_void_p()
    props = PoolProps(allocType=1, locationType=1, locationId=0, maxSize=limit)
    assert cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
    assert cu.cuDeviceGetMemPool(ctypes.byref(usual), 0) == 0
    assert cu.cuDeviceSetMemPool(0, pool) == 0

    def used(attr=USED_MEM_CURRENT):
        torch.cuda.synchronize()
        x = ctypes.c_uint64()
        assert cu.cuMemPoolGetAttribute(pool, attr, ctypes.byref(x)) == 0
        return x.value

    try:
        yield used
    finally:
        torch.cuda.synchronize()
        assert cu.cuDeviceSetMemPool(0, usual) == 0


def test_a_reported_failure_is_not_reported_again(pvt):
    """A call refused for want of memory leaves no error behind: the thread's
    next call, of this library or of torch, does not fail with it."""
    import torch
    rp, col = mesh(1400, 1400)
    with limited_pool(32 << 20):
        with pytest.raises(pvt.PivoterError) as e:
            gpu_dag(pvt, rp, col, validate=False)
        assert e.value.status == 3
        assert int(torch.zeros(4, device="cuda").sum()) == 0
    dag = gpu_dag(pvt, rp, col, validate=False)
    assert pvt.to_ints(dag.count_global(kmax=4)) == [0, 1400 * 1400, len(col) // 2, 0, 0]
    dag.free()


def test_an_orientation_that_finds_no_room_leaves_nothing_behind(pvt):
    """A mesh, which takes the core rounds and then the level-wise peel, with
    ever more room: each orientation is refused or right, and none keeps memory."""
    rp, col = mesh(1400, 1400)
    ends = set()
    for limit in range(32 << 20, 400 << 20, 16 << 20):
        with limited_pool(limit) as used:
            try:
                dag = gpu_dag(pvt, rp, col, validate=False)
            except pvt.PivoterError as e:
                assert e.status == 3
                ends.add("refused")
            else:
                assert dag.alpha == 2 and int((dag.cores() != 2).sum()) == 0
                dag.free()
                ends.add("oriented")
            assert used() == 0
        if "oriented" in ends:
            break
    assert ends == {"refused", "oriented"}


def test_a_refused_count_leaves_nothing_in_flight(pvt):
    """Per-edge counts launch the widest class first.  Where a narrower one then
    finds no room, the call returns with every launched class finished: the
    table it was given does not change any more."""
    import torch
    rp, col = graphgen.generate(4000, er_avg_deg=8.0, planted=[(12, 100, 120, 0.75), (8, 40, 60, 0.8)], seed=53)
    dag = gpu_dag(pvt, rp, col)
    want = dag.count_local_edge(kmax=4)
    dag.free()
    peek = torch.cuda.Stream()
    refused = 0
    for limit in range(32 << 20, 640 << 20, 32 << 20):
        dag = gpu_dag(pvt, rp, col)
        out = torch.empty_like(want)
        torch.cuda.synchronize()
        with limited_pool(limit):
            try:
                dag.count_local_edge(kmax=4, out=out)
            except pvt.PivoterError as e:
                assert e.status == 3
                refused += 1
                with torch.cuda.stream(peek):
                    now = out.clone()
                torch.cuda.synchronize()
                assert torch.equal(now, out)
                done = False
            else:
                assert torch.equal(out, want)
                done = True
        dag.free()
        if done:
            break
    assert refused > 0 and done


def test_tables_of_a_refused_count_are_built_anew(pvt):
    """A count that finds no room for its edge ids or its Pascal table is
    refused, and the next one, with room, does not take them for built."""
    import torch
    rp, col = graphgen.generate(2_000_000, er_avg_deg=6.0, planted=[(2, 20, 40, 0.9)], seed=52)
    ref = oracle.count(rp, col, kmax=6)
    K = 6
    dag = gpu_dag(pvt, rp, col)
    want = [dag.count_local_edge(kmax=4), dag.count_global(kmax=K)]
    assert pvt.to_ints(want[1]) == ref["C"]
    dag.free()
    refused = 0
    for limit in range(32 << 20, 160 << 20, 32 << 20):
        dag = gpu_dag(pvt, rp, col)
        out = torch.empty_like(want[0])
        with limited_pool(limit):
            for call in (lambda: dag.count_local_edge(kmax=4, out=out), lambda: dag.count_global(kmax=K, W=18)):
                try:
                    call()
                except pvt.PivoterError as e:
                    assert e.status == 3
                    refused += 1
        assert torch.equal(dag.count_local_edge(kmax=4, out=out), want[0])
        assert torch.equal(dag.count_global(kmax=K), want[1])
        dag.free()
    assert refused > 0


def classes_graph():
    """Roots of every class up to 512: 40,000 of at most 32 out-neighbours, and
    dense groups whose roots are split, walked by blocks and walked in parts."""
    return disjoint(graphgen.generate(40_000, er_avg_deg=9.0, planted=[(30, 24, 30, 0.8), (12, 40, 60, 0.7),
                                                                       (4, 90, 120, 0.5)], seed=54),
                    graphs.clique_minus_random(180, 9, 55), graphs.clique_minus_random(300, 9, 56))


COUNTS = {
    "global": lambda dag, K: dag.count_global(kmax=K),
    "range": lambda dag, K: dag.combine_hist(dag.count_hist(0, dag.n, kmax=K), kmax=K),
    "vertex": lambda dag, K: dag.count_local_vertex(kmax=3),
    "edge": lambda dag, K: dag.count_local_edge(kmax=3),
}


@pytest.mark.parametrize("what", sorted(COUNTS))
def test_counts_within_a_scratch_limit(pvt, what):
    """Under any limit the counts, and the tree that is walked, are those of the
    call without one: with frames for some of the roots, the gather in passes,
    dense roots walked where they are met, and nothing optional at all."""
    import torch
    rp, col = classes_graph()
    dag = gpu_dag(pvt, rp, col)
    assert dag.alpha > 256
    want = COUNTS[what](dag, 4)
    ref = oracle.count(rp, col, kmax=4)
    if want.dim() == 2:
        assert pvt.to_ints(want) == ref["C"]
    tree = [dag.stats()[k] for k in ("sct_nodes", "sct_leaves", "pivot_words", "roots")]
    launches = {}
    for mb in [1, *range(48, 321, 8), 0]:
        dag.set_scratch_limit(mb << 20)
        assert torch.equal(COUNTS[what](dag, 4), want), mb
        st = dag.stats()
        if what in ("global", "vertex", "edge"):
            assert [st[k] for k in ("sct_nodes", "sct_leaves", "pivot_words", "roots")] == tree, mb
        launches[mb] = st["launches"]
    if what == "global":
        assert max(launches.values()) > launches[0]  # the gather went in passes
    if what != "range":  # (whose last call is the combine)
        assert min(launches.values()) < launches[0]  # something optional was left out
    dag.free()


@pytest.mark.parametrize("what", sorted(COUNTS))
def test_a_count_fits_where_its_required_scratch_does(pvt, what):
    """Optional buffers take what the required ones leave: in the memory that a
    count needs without any, it is not refused."""
    import torch
    rp, col = classes_graph()
    dag = gpu_dag(pvt, rp, col)
    want = COUNTS[what](dag, 4)
    dag.free()
    dag = gpu_dag(pvt, rp, col)
    dag.set_scratch_limit(1)
    with limited_pool(1 << 40) as used:
        assert torch.equal(COUNTS[what](dag, 4), want)
        need = used(RESERVED_MEM_HIGH)
    dag.free()
    dag = gpu_dag(pvt, rp, col)
    with limited_pool(need):
        assert torch.equal(COUNTS[what](dag, 4), want)
        # ... nor is another count on the dag, whose optional buffers the first one's are
        for other in sorted(COUNTS):
            try:
                COUNTS[other](dag, 4)
            except pvt.PivoterError as e:
                assert e.status == 3
        assert torch.equal(COUNTS[what](dag, 4), want)
    dag.free()


def test_a_recorded_count_after_its_frames_moved(pvt):
    """A recorded count whose frames another call has since moved to less room is
    recorded anew, whatever the address."""
    import torch
    rp, col = classes_graph()
    dag = gpu_dag(pvt, rp, col)
    want = dag.count_global(kmax=5)
    dag.set_policy(graph=True)
    out = torch.empty_like(want)
    for limit in (1 << 40, 256 << 20, 224 << 20, 192 << 20, 1 << 40):
        with limited_pool(limit):
            for _ in range(3):
                assert torch.equal(dag.count_global(kmax=5, out=out.zero_()), want)
            dag.set_scratch_limit(0)  # the frames move
            dag.count_hist(0, dag.n, kmax=5)
            assert torch.equal(dag.count_global(kmax=5, out=out.zero_()), want)
    dag.free()


@pytest.mark.parametrize("kind", ["global", "vertex", "edge"])
def test_a_direct_query_keeps_to_the_budget(pvt, kind):
    """A server's direct query takes no more device memory than the budget holds
    for it: optional buffers come out of what was reserved."""
    rp, col = classes_graph()
    dag = gpu_dag(pvt, rp, col)
    want = {"global": dag.count_global, "vertex": dag.count_local_vertex, "edge": dag.count_local_edge}[kind](kmax=3)
    dag.free()
    budget = 512 << 20
    with limited_pool(1 << 40) as used:
        with pvt.Server(mem_budget=budget, direct_edges=1) as sv:
            t = sv.submit(rp, col, kind, kmax=3)
            assert sv.wait(t, 60000)
            got = sv.result(t)[0].view(np.int64)
        assert used(RESERVED_MEM_HIGH) <= budget
    assert np.array_equal(got.reshape(-1), want.cpu().numpy().reshape(-1))


def test_a_batch_keeps_to_the_budget(pvt):
    """Batched per-edge counts of dense graphs take their tables out of what the
    budget has left, and fewer warps walk where that is little."""
    qs = [graphs.gnp(110 + i, 0.5, 60 + i) for i in range(8)] + [graphs.gnp(60 + i, 0.5, 70 + i) for i in range(8)]
    want = []
    for rp, col in qs:
        dag = gpu_dag(pvt, rp, col)
        want.append(dag.count_local_edge(kmax=4).cpu().numpy().reshape(-1))
        dag.free()
    for budget in (16 << 20, 64 << 20, 4 << 30):
        with limited_pool(max(budget, 32 << 20)) as used:
            with pvt.Server(mem_budget=budget, direct_edges=-1) as sv:
                tickets = [sv.submit(rp, col, "edge", kmax=4) for rp, col in qs]
                got = []
                for t in tickets:
                    assert sv.wait(t, 60000)
                    got.append(sv.result(t)[0].view(np.int64).reshape(-1))
            assert used(RESERVED_MEM_HIGH) <= max(budget, 32 << 20)
        assert all(np.array_equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("extra", ["into the core", "out of the core"])
def test_an_asymmetric_csr_is_refused_before_its_out_lists_are_written(pvt, extra):
    """K_40 and 20 more vertices with 400 arcs one way.  Trusted without
    validation, its out-lists would have more entries than nnz / 2 (arcs from
    vertices that come before the core), or fewer."""
    rows = [[u for u in range(40) if u != v] for v in range(40)] + [[] for _ in range(20)]
    for v in range(40, 60):
        for u in range(20):
            (rows[v] if extra == "into the core" else rows[u]).append(u if extra == "into the core" else v)
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    col = np.concatenate([np.asarray(r, np.uint32) for r in rows])
    with pytest.raises(pvt.PivoterError) as e:
        gpu_dag(pvt, rp, col, validate=False)
    assert e.value.status == 2


def test_large_frames_go_back_to_the_device(pvt):
    """A dag whose frame buffer passed 6 GiB leaves at most that, beyond what is
    in use, in the device's pool."""
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    pool = ctypes.c_void_p()

    def held(attr):
        torch.cuda.synchronize()
        x = ctypes.c_uint64()
        assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
        assert cu.cuMemPoolGetAttribute(pool, attr, ctypes.byref(x)) == 0
        return x.value

    rp, col = disjoint(*[graphs.clique_minus_random(1000, 9, 57 + i) for i in range(4)])
    dag = gpu_dag(pvt, rp, col)
    before = held(USED_MEM_CURRENT)
    dag.count_global(kmax=4)
    assert held(USED_MEM_CURRENT) - before > 6 << 30
    dag.free()
    assert held(RESERVED_MEM_CURRENT) - held(USED_MEM_CURRENT) <= 6 << 30


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
