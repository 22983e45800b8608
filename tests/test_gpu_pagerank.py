"""GPU parity of dynamic PageRank (sp_pr_*) against the single-precision
oracle (appendix listing "Dynamic PR").

Ranks are compared with a tolerance: a vertex with at most eight in-edges is
summed in in-neighbour order, as the oracle does, but larger in-lists are
summed in parallel parts whose float rounding differs; the difference stays
within a few units in the last place of the sums and is damped by the
factor d < 1 through later steps.  The batch counters, the flagged-vertex
counts and the edge sets must match exactly, and the number of Jacobi
steps may differ by at most one (a step whose difference lies within
rounding of beta)."""
import numpy as np
import pytest

import oracle
from paper_2507_11094_gb300 import sp
from paper_2507_11094_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
D, BETA, ITERS = 0.85, 1e-6, 100
RTOL, ATOL = 2e-5, 1e-9


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2507_11094_gb300 import build
    build.build()
    oracle.build()
    sp.load()


WORKLOADS = {
    "er1k": lambda: wl.tiny_er(4),
    "rmat12": lambda: wl.rmat(12, batch_frac=0.01, seed=3),
    "grid48": lambda: wl.grid(48, 48, batch_frac=0.01, seed=2, tree_fraction=0.0),
}


@pytest.mark.parametrize("name", list(WORKLOADS))
def test_static_pagerank(name):
    W = WORKLOADS[name]()
    ref = oracle.OracleGraph(W.n, W.row_off, W.col, W.w)
    want, it = ref.pagerank(D, BETA, ITERS)
    with sp.Graph(W.n, W.row_off, W.col, W.w) as g:
        st = g.pr_init(D, BETA, ITERS, stats=True)
        got = g.pr_get()
    np.testing.assert_allclose(got, want, rtol=RTOL, atol=ATOL)
    assert abs(st.rounds_push - it) <= 1
    assert st.relaxed_edges == W.m * st.rounds_push


@pytest.mark.parametrize("name", list(WORKLOADS))
def test_dynamic_pagerank_batches(name):
    W = WORKLOADS[name]()
    ref = oracle.OracleGraph(W.n, W.row_off, W.col, W.w)
    want, _ = ref.pagerank(D, BETA, ITERS)
    with sp.Graph(W.n, W.row_off, W.col, W.w) as g:
        g.pr_init(D, BETA, ITERS)
        for k in range(4):
            b = W.batch(k)
            cnt = ref.pagerank_batch(b, want, D, BETA, ITERS)
            st = g.pr_apply(b, stats=True)
            assert (st.n_del_applied, st.n_del_absent, st.n_add_applied,
                    st.n_add_present) == cnt[:4]
            assert st.affected == cnt[4] + cnt[5]
            assert abs(st.rounds_push - (cnt[6] + cnt[7])) <= 2
            np.testing.assert_allclose(g.pr_get(), want, rtol=RTOL, atol=ATOL)
            for x, y in zip(g.export_csr(), ref.csr()):
                np.testing.assert_array_equal(x, y)


def reach(n, ro, col, seeds):
    from scipy.sparse import csr_matrix
    from scipy.sparse.csgraph import breadth_first_order
    A = csr_matrix((np.ones(col.size), col, ro), shape=(n, n))
    seen = np.zeros(n, bool)
    for s in np.unique(seeds):
        if not seen[s]:
            seen[breadth_first_order(A, int(s), directed=True,
                                     return_predecessors=False)] = True
    return seen


def test_unflagged_vertices_keep_their_ranks_exactly():
    # a sparse graph with many vertices unreachable from the updates
    n = 3000
    ro, col, w = wl.er_digraph(n, 4500, 1, 9, 11)
    stream = wl.BatchStream(n, ro, col, w, 1, 9, "uniform")
    with sp.Graph(n, ro, col, w) as g:
        g.pr_init(D, BETA, ITERS)
        before = g.pr_get()
        b = stream.next(3, 3, seed=5)
        h = oracle.OracleGraph(n, ro, col, w)
        flagged = reach(n, ro, col, b.del_dst)
        z = np.zeros(0, np.int32)
        h.apply_batch(b.del_src, b.del_dst, z, z, z)
        r1, c1, _ = h.csr()
        flagged |= reach(n, r1, c1, b.add_dst)
        st = g.pr_apply(b, stats=True)
        after = g.pr_get()
        assert 0 < flagged.sum() < n
        assert st.affected <= 2 * flagged.sum()
        np.testing.assert_array_equal(after[~flagged], before[~flagged])


def test_empty_and_invalid_batches():
    W = wl.tiny_er(5)
    with sp.Graph(W.n, W.row_off, W.col, W.w) as g:
        g.pr_init(D, BETA, ITERS)
        before = g.pr_get()
        z = np.zeros(0, np.int32)
        st = g.pr_apply_batch(z, z, z, z, z, stats=True)
        assert st.affected == 0
        np.testing.assert_array_equal(g.pr_get(), before)
        m = g.m
        with pytest.raises(sp.SpError) as e:   # the bad insertion is in phase two
            g.pr_apply_batch(np.array([0], np.int32), np.array([1], np.int32),
                             np.array([0], np.int32), np.array([W.n], np.int32),
                             np.array([3], np.int32))
        assert e.value.code == sp.SP_EINVAL
        assert g.m == m
        np.testing.assert_array_equal(g.pr_get(), before)


def test_pagerank_and_sssp_states():
    W = wl.tiny_er(6)
    with sp.Graph(W.n, W.row_off, W.col, W.w) as g:
        with pytest.raises(sp.SpError) as e:
            g.pr_get()
        assert e.value.code == sp.SP_ESTATE
        g.sssp_init(W.source)
        g.pr_init(D, BETA, ITERS)
        g.get_dist()                         # static PR leaves distances valid
        g.pr_apply(W.batch(0))
        with pytest.raises(sp.SpError) as e:
            g.get_dist()
        assert e.value.code == sp.SP_ESTATE
        g.sssp_init(W.source)
        ref = oracle.OracleGraph(W.n, *g.export_csr())
        np.testing.assert_array_equal(g.get_dist(), ref.dijkstra(W.source))
        g.apply(W.batch(1))
        with pytest.raises(sp.SpError) as e:
            g.pr_get()
        assert e.value.code == sp.SP_ESTATE
        with pytest.raises(sp.SpError):
            g.pr_init(1.5, BETA, ITERS)


def ranks64(n, u, v, iters):
    """`iters` Jacobi steps over every vertex, in 64 bits (with the 32-bit
    damping the call takes)."""
    d = float(np.float32(D))
    od = np.bincount(u, minlength=n).astype(np.float64)
    pr = np.full(n, 1.0 / n)
    for _ in range(iters):
        term = np.divide(pr, od, out=np.zeros(n), where=od > 0)
        pr = (1.0 - d) / n + d * np.bincount(v, weights=term[u], minlength=n)
    return pr


# Rows at the bounds of the in-degree classes (a lane's 8, a group's 64, a
# warp's 1,024, and cut into one to six segments), more vertices than terms in
# shared memory, and out-degrees that fill those in part, exactly by one
# out-degree bin, or not at all.  Each step rounds a sum of terms over a tree
# (at most eight 4-term words a lane, five levels, six parts: under 32 units
# of 2^-24), and later steps damp it by d: under 32 / (1 - d) * 2^-24 = 1.3e-5.
@pytest.mark.parametrize("n,extra", [(3000, 0), (7001, 20000), (60000, 150000), (200000, 0),
                                     (200000, 700000)])
def test_rows_of_every_class(n, extra):
    rng = np.random.default_rng(n + extra)
    degs = [1, 3, 4, 5, 8, 9, 31, 32, 33, 63, 64, 65, 127, 128, 129, 1023, 1024, 1025, 2047, 2048,
            2049, 2999] + ([6000, 6145] if n > 6200 else [])
    keys = [rng.choice(n - 1, size=d, replace=False) for d in degs]
    u = np.concatenate([np.where(k >= 7 * i, k + 1, k) for i, k in enumerate(keys)])
    v = np.repeat(7 * np.arange(len(degs)), degs)
    u = np.concatenate([u, rng.integers(0, n, extra)])
    v = np.concatenate([v, rng.integers(0, n, extra)])
    key = np.unique(u.astype(np.int64) * n + v)
    u, v = key // n, key % n
    ro = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(u, minlength=n), out=ro[1:])
    with sp.Graph(n, ro, v.astype(np.int32), np.ones(v.size, np.int32)) as g:
        for iters in (1, 2, 9):
            st = g.pr_init(D, 0.0, iters, stats=True)
            assert st.rounds_push <= iters and st.relaxed_edges == v.size * st.rounds_push
            np.testing.assert_allclose(g.pr_get(), ranks64(n, u, v, iters), rtol=2e-5)
        # the same ranks bit for bit: a step's sums do not depend on the schedule
        a = g.pr_get()
        g.pr_init(D, 0.0, 9)
        np.testing.assert_array_equal(g.pr_get(), a)


def test_lists_without_memory_of_their_own():
    # the packed in-neighbour lists do not fit: they go to the store's
    # alternate regions, with the same ranks, and batches keep working
    W = wl.rmat(12, batch_frac=0.02, seed=8)
    state = {"refuse": False, "refused": 0}

    def refuse(nbytes):
        if state["refuse"] and nbytes >= 4 * W.m:
            state["refused"] += 1
            return True
        return False
    with sp.Graph(W.n, W.row_off, W.col, W.w) as g:
        g.pr_init(D, BETA, ITERS)
        want = g.pr_get()
        b = W.batch(0)
        g.pr_apply(b)
        after = g.pr_get()
    with sp.Graph(W.n, W.row_off, W.col, W.w, refuse_alloc=refuse) as g:
        g.reserve(4096)
        state["refuse"] = True
        g.pr_init(D, BETA, ITERS)
        assert state["refused"] > 0
        np.testing.assert_array_equal(g.pr_get(), want)
        g.pr_apply(b)
        np.testing.assert_array_equal(g.pr_get(), after)
        state["refuse"] = False
        ref = oracle.OracleGraph(W.n, W.row_off, W.col, W.w)
        ref.apply(b)
        for x, y in zip(g.export_csr(), ref.csr()):
            np.testing.assert_array_equal(x, y)


def test_vertices_without_edges_are_passed_over_quickly():
    # 10 M vertices, most of them without in-edges: what a step does for those
    # (in the first two only) is short beside a launch's preparation (two steps
    # took 1.5 times as long as one when each of their rows waited for memory alone)
    import time
    n, m = 10 ** 7, 10 ** 6
    key = np.unique(np.random.default_rng(1).integers(0, n * n, m))
    ro = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(key // n, minlength=n), out=ro[1:])
    best = {}
    with sp.Graph(n, ro, (key % n).astype(np.int32), np.ones(key.size, np.int32)) as g:
        for iters in (1, 2):
            times = []
            for _ in range(8):
                t0 = time.perf_counter()
                g.pr_init(D, 0.0, iters)
                times.append(time.perf_counter() - t0)
            best[iters] = min(times)
            np.testing.assert_allclose(g.pr_get(), ranks64(n, key // n, key % n, iters), rtol=2e-5)
    assert best[2] < 1.35 * best[1], best
