"""GPU tests of calls on a handle whose edge count on the host lags behind the
stores (an asynchronous batch that nobody has finished, a phase that ran into
a bound): results follow the stores' rows, whatever the host believes."""
import numpy as np
import pytest

import oracle
from paper_2507_11094_gb300 import sp
from paper_2507_11094_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2507_11094_gb300 import build
    build.build()
    oracle.build()
    sp.load()


def insertions(n, keys, w):
    i32 = lambda x: np.ascontiguousarray(x, np.int32)
    z = np.zeros(0, np.int32)
    return wl.Batch(z, z, i32(keys // n), i32(keys % n), i32(w))


def launch_unfinished(g, b):
    """Apply b asynchronously; the host is never told the outcome."""
    import torch
    x = g.capture(*[torch.from_numpy(a).cuda() for a in
                    (b.del_src, b.del_dst, b.add_src, b.add_dst, b.add_w)])
    x.launch()
    g.sync()
    return x


# new edges whose in-neighbour lists take several times the room that the
# host's count asks for, and just more than it
@pytest.mark.parametrize("n,m,k", [(120, 1000, 6000), (1000, 4000, 12000), (100, 5000, 2500),
                                   (3000, 20000, 9000)])
def test_ranks_of_a_graph_with_more_edges_than_the_host_knows(n, m, k):
    import torch
    ro, col, w = wl.er_digraph(n, m, 1, 100, seed=n)
    ref = oracle.OracleGraph(n, ro, col, w)
    rng = np.random.default_rng(m)
    free = np.setdiff1d(np.arange(n * n), wl.csr_keys(n, ro, col))
    b = insertions(n, rng.choice(free, size=k, replace=False), rng.integers(1, 101, k))
    with sp.Graph(n, ro, col, w, stream=torch.cuda.Stream()) as g:
        g.sssp_init(0)
        g.reserve(k)
        x = launch_unfinished(g, b)
        ref.apply(b)
        np.testing.assert_array_equal(g.get_dist(), ref.dijkstra(0))   # it applied
        assert g.m == m
        st = g.pr_init(0.85, 1e-6, 100, stats=True)
        want, it = ref.pagerank(0.85, 1e-6, 100)
        # (the bounds of the ranks' own parity tests)
        np.testing.assert_allclose(g.pr_get(), want, rtol=2e-5, atol=1e-9)
        assert abs(st.rounds_push - it) <= 1
        assert st.relaxed_edges == (m + k) * st.rounds_push
        x.close()


def test_triangles_of_hubs_that_the_host_does_not_know():
    # an empty graph becomes three hubs, joined to each other and to every vertex
    # of a rim: rows that the whole grid orients (more than 65,536 entries), and
    # the hubs' own triangle is counted from such a row.  Nobody finishes the batch
    import torch
    k = 66000
    hubs = np.array([7, 30000, 66002], np.int64)
    rim = np.setdiff1d(np.arange(k + 3), hubs)
    n = 200000                       # (with room in the spare pool for the hubs' rows)
    u = np.concatenate([np.repeat(hubs, k), [7, 7, 30000]])
    v = np.concatenate([np.tile(rim, 3), [30000, 66002, 66002]])
    u, v = np.concatenate([u, v]), np.concatenate([v, u])
    b = insertions(n, u * n + v, np.ones(u.size, np.int64))
    z = np.zeros(0, np.int32)
    with sp.Graph(n, np.zeros(n + 1, np.int64), z, z, slack=0.0,
                  stream=torch.cuda.Stream()) as g:
        g.sssp_init(0)
        g.reserve(u.size)
        x = launch_unfinished(g, b)
        assert g.m == 0
        assert g.get_dist()[:k + 3].max() == 2   # it applied: all are two steps apart at most
        assert g.tc_init() == 3 * k + 1
        x.close()


# a rank batch of which a phase's flags run into a round cap: the phase's edges
# are merged, so the edge count follows, what held on the old edges no longer
# does, and the ranks can be computed again (also through one block's plan)
@pytest.mark.parametrize("nd,na", [(0, 2500), (0, 700), (1500, 0), (600, 2500)])
def test_a_rank_batch_that_hits_a_bound_leaves_the_edge_count_right(nd, na):
    n, m = 100, 5000
    ro, col, w = wl.er_digraph(n, m, 1, 100, seed=7)
    keys = wl.csr_keys(n, ro, col)
    rng = np.random.default_rng(nd + na)
    gone = rng.choice(keys, size=nd, replace=False)
    new = rng.choice(np.setdiff1d(np.arange(n * n), keys), size=na, replace=False)
    i32 = lambda x: np.ascontiguousarray(x, np.int32)
    b = wl.Batch(i32(gone // n), i32(gone % n), i32(new // n), i32(new % n),
                 i32(rng.integers(1, 101, na)))
    # the first phase that has updates hits the bound, and the call ends there
    z = np.zeros(0, np.int32)
    done = b if not nd else wl.Batch(b.del_src, b.del_dst, z, z, z)
    ref = oracle.OracleGraph(n, ro, col, w)
    with sp.Graph(n, ro, col, w) as g:
        g.sssp_init(0)
        g.pr_init(0.85, 1e-6, 100)
        g.set_limits(1)
        with pytest.raises(sp.SpError) as e:
            g.pr_apply(b)
        assert e.value.code == sp.SP_ETIMEOUT
        g.set_limits(0)
        ref.apply(done)
        assert g.m == m - done.del_src.size + done.add_src.size
        for call in (g.get_dist, g.pr_get):
            with pytest.raises(sp.SpError) as e:
                call()
            assert e.value.code == sp.SP_ESTATE
        for rev in (False, True):
            got = g.export_csr(reverse=rev)
            rro, rcol, rw = ref.csr()
            u = np.repeat(np.arange(n), np.diff(rro))
            if rev:
                order = np.lexsort((u, rcol))
                want = (np.concatenate([[0], np.cumsum(np.bincount(rcol, minlength=n))]),
                        u[order], rw[order])
            else:
                want = (rro, rcol, rw)
            for x, y in zip(got, want):
                np.testing.assert_array_equal(x, y)
        g.pr_init(0.85, 1e-6, 100)
        np.testing.assert_allclose(g.pr_get(), ref.pagerank(0.85, 1e-6, 100)[0], rtol=2e-5,
                                   atol=1e-9)
        g.sssp_init(0)
        np.testing.assert_array_equal(g.get_dist(), ref.dijkstra(0))
