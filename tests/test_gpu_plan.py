"""GPU tests of small batches, whose store update one block plans, around the
largest one (1,024 updates, above which the grid's sort and count take over)
and at odd and tiny sizes: counters, both stores and distances against the
oracle, with repeated updates, no-ops and delete-then-insert among them."""
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


def messy(rng, n, keys, k):
    """k updates: deletions of present and absent edges and insertions of new
    and present ones, a third of them repeated (insertions with other weights)
    or naming an edge that the batch deletes too."""
    nd = int(rng.integers(0, k + 1)) if k > 1 else int(rng.integers(0, 2))
    na = k - nd

    def some(count):
        pick = rng.choice(keys, size=count)
        rnd = rng.integers(0, n * n, size=count)
        return np.where(rng.random(count) < 0.6, pick, rnd)
    d, a = some(nd), some(na)
    for x in (d, a):
        if x.size > 2:
            again = rng.random(x.size) < 0.3
            x[again] = rng.choice(x, size=int(again.sum()))
    if nd and na:
        both = rng.random(na) < 0.2
        a[both] = rng.choice(d, size=int(both.sum()))
    w = rng.integers(1, 101, size=na)
    i32 = lambda x: np.ascontiguousarray(x, np.int32)
    return wl.Batch(i32(d // n), i32(d % n), i32(a // n), i32(a % n), i32(w))


@pytest.mark.parametrize("n,m", [(40, 300), (5000, 40000)])
@pytest.mark.parametrize("sizes", [(1, 1, 1, 2, 3), (31, 32, 33, 64, 65), (511, 512, 513, 700, 700),
                                   (1022, 1023, 1024, 1025, 1026), (1024, 1024, 1024, 1100, 1)])
@pytest.mark.parametrize("own_stream", [False, True])
def test_small_batches(n, m, sizes, own_stream):
    import torch
    ro, col, w = wl.er_digraph(n, m, 1, 100, seed=n)
    ref = oracle.OracleGraph(n, ro, col, w)
    rng = np.random.default_rng(n + sizes[0])
    st = torch.cuda.Stream() if own_stream else None
    with sp.Graph(n, ro, col, w, slack=0.05, stream=st) as g:
        g.sssp_init(0)
        for k in sizes:
            ro, col, _ = ref.csr()
            b = messy(rng, n, wl.csr_keys(n, ro, col), k)
            want = ref.apply(b)
            got = g.apply(b, stats=True)
            assert (got.n_del_applied, got.n_del_absent, got.n_add_applied,
                    got.n_add_present) == want
            np.testing.assert_array_equal(g.get_dist(), ref.dijkstra(0))
            for x, y in zip(g.export_csr(), ref.csr()):
                np.testing.assert_array_equal(x, y)
        ro, col, w = ref.csr()
        u = np.repeat(np.arange(n), np.diff(ro))
        order = np.lexsort((u, col))
        rro, rcol, rw = g.export_csr(reverse=True)
        np.testing.assert_array_equal(np.diff(rro), np.bincount(col, minlength=n))
        np.testing.assert_array_equal(rcol, u[order])
        np.testing.assert_array_equal(rw, w[order])


@pytest.mark.parametrize("k", [1, 7, 1024])
def test_an_invalid_update_changes_nothing(k):
    n = 300
    ro, col, w = wl.er_digraph(n, 2000, 1, 100, seed=3)
    with sp.Graph(n, ro, col, w) as g:
        g.sssp_init(0)
        before = g.get_dist()
        z = np.zeros(0, np.int32)
        for bad in ((k - 1, n, 1), (0, -1, 1), (k // 2, 5, 0), (k // 2, 5, sp.SP_WMAX + 1)):
            d = np.full(k, 7, np.int32)
            ww = np.ones(k, np.int32)
            d[bad[0]], ww[bad[0]] = bad[1], bad[2]
            with pytest.raises(sp.SpError) as e:
                g.apply_batch(z, z, np.arange(k, dtype=np.int32) % n, d, ww)
            assert e.value.code == sp.SP_EINVAL
        np.testing.assert_array_equal(g.get_dist(), before)
        for x, y in zip(g.export_csr(), (ro, col, w)):
            np.testing.assert_array_equal(x, y)


# distances through the handle's page-locked block and, above 16,384 vertices,
# through a device buffer; batches read in place from pageable and page-locked
# arrays, and one update more
@pytest.mark.parametrize("n", [1, 3, 16383, 16384, 16385])
@pytest.mark.parametrize("pinned", [False, True])
def test_small_host_arrays(n, pinned):
    import torch

    def host(x):
        if not pinned or not x.size:
            return x
        t = torch.empty(x.size, dtype=torch.int32, pin_memory=True)
        t.numpy()[:] = x
        return t.numpy()
    m = min(4 * n, n * (n - 1))
    ro, col, w = wl.er_digraph(n, m, 1, 100, seed=n) if m else (np.zeros(n + 1, np.int64),
                                                                 np.zeros(0, np.int32),
                                                                 np.zeros(0, np.int32))
    ref = oracle.OracleGraph(n, ro, col, w)
    rng = np.random.default_rng(n)
    from oracle.invariants import check_sssp
    with sp.Graph(n, ro, col, w, stream=torch.cuda.Stream()) as g:
        g.sssp_init(0)
        for k in (5, 5, 5, 1024, 1025):
            if n == 1:
                break
            ro, col, _ = ref.csr()
            keys = wl.csr_keys(n, ro, col) if col.size else np.array([1])
            b = messy(rng, n, keys, k)
            ref.apply(b)
            d, p = np.full(n, -7, np.int32), np.full(n, -7, np.int32)
            a = [host(x) for x in (b.del_src, b.del_dst, b.add_src, b.add_dst, b.add_w)]
            g.apply_batch_get(*a, dist=d, parent=p)
            np.testing.assert_array_equal(d, ref.dijkstra(0))
            check_sssp(n, *ref.csr(), 0, d, p)
        d, p = g.get_dist(parent=True)
        np.testing.assert_array_equal(d, ref.dijkstra(0))
        check_sssp(n, *ref.csr(), 0, d, p)


@pytest.mark.parametrize("n,m", [(600, 5000), (5000, 40000), (300000, 500000)])
@pytest.mark.parametrize("blocks", [0, 1, 3])
def test_grid_sorted_batches(n, m, blocks):
    """Batches just above what one block plans and around whole tiles of the
    grid's sort, either store in half of its blocks (or both in one block),
    with the ids that take digits of ten bits and of nine."""
    ro, col, w = wl.er_digraph(n, m, 1, 100, seed=n)
    ref = oracle.OracleGraph(n, ro, col, w)
    rng = np.random.default_rng(n + blocks)
    with sp.Graph(n, ro, col, w, slack=0.05) as g:
        if blocks:
            g.set_loop_blocks(blocks)
        g.sssp_init(0)
        for k in (1025, 2048, 2049, 4096, 4097, 8193, 20001):
            ro, col, _ = ref.csr()
            b = messy(rng, n, wl.csr_keys(n, ro, col), k)
            want = ref.apply(b)
            got = g.apply(b, stats=True)
            assert (got.n_del_applied, got.n_del_absent, got.n_add_applied,
                    got.n_add_present) == want
            for x, y in zip(g.export_csr(), ref.csr()):
                np.testing.assert_array_equal(x, y)
        np.testing.assert_array_equal(g.get_dist(), ref.dijkstra(0))
        ro, col, w = ref.csr()
        u = np.repeat(np.arange(n), np.diff(ro))
        order = np.lexsort((u, col))
        rro, rcol, rw = g.export_csr(reverse=True)
        np.testing.assert_array_equal(np.diff(rro), np.bincount(col, minlength=n))
        np.testing.assert_array_equal(rcol, u[order])
        np.testing.assert_array_equal(rw, w[order])


# above one block's batches the old-row searches run beside the sort, on the
# handle's side stream (none on the legacy stream); only then are they read
@pytest.mark.parametrize("own_stream", [False, True])
def test_searches_beside_the_sort_of_triangle_and_rank_batches(own_stream):
    import torch
    st = torch.cuda.Stream() if own_stream else None
    W = wl.sym_er(4096, 40000, 700, 3)       # 2,800 updates a batch
    ref = oracle.OracleGraph(W.n, W.row_off, W.col, W.w)
    with sp.Graph(W.n, W.row_off, W.col, W.w, stream=st) as g:
        assert g.tc_init() == ref.triangles()
        for k in range(4):
            b = W.batch(k)
            cnt = ref.apply(b)
            c, s = g.tc_apply(b, stats=True)
            assert (s.n_del_applied, s.n_del_absent, s.n_add_applied, s.n_add_present) == cnt
            assert c == ref.triangles()
    W = wl.rmat(13, batch_frac=0.04, seed=3)   # two phases of 2,600 updates
    ref = oracle.OracleGraph(W.n, W.row_off, W.col, W.w)
    want, _ = ref.pagerank(0.85, 1e-6, 100)
    with sp.Graph(W.n, W.row_off, W.col, W.w, stream=st) as g:
        g.pr_init(0.85, 1e-6, 100)
        for k in range(4):
            b = W.batch(k)
            assert min(b.del_src.size, b.add_src.size) > 1024
            cnt = ref.pagerank_batch(b, want, 0.85, 1e-6, 100)
            s = g.pr_apply(b, stats=True)
            assert (s.n_del_applied, s.n_del_absent, s.n_add_applied, s.n_add_present) == cnt[:4]
            # (the bounds of the ranks' own parity tests)
            np.testing.assert_allclose(g.pr_get(), want, rtol=2e-5, atol=1e-9)
            for x, y in zip(g.export_csr(), ref.csr()):
                np.testing.assert_array_equal(x, y)


def test_one_update_of_a_hub_merges_as_fast_as_many():
    # the hub's row is 7,800 strips of the merge whatever the batch's size; seven
    # hundred updates start the whole grid (with a block per item only, one
    # update's merge took the time of two blocks: tens of times as long)
    n = 2000003
    ro = np.concatenate([[0], np.full(n, n - 1)]).astype(np.int64)
    col = np.arange(1, n, dtype=np.int32)
    z = np.zeros(0, np.int32)
    best = {}
    with sp.Graph(n, ro, col, np.ones(n - 1, np.int32)) as g:
        g.sssp_init(0)
        for k in (1, 700):
            d = (np.arange(k, dtype=np.int32) * 2801 + 17).astype(np.int32)
            o = np.zeros(k, np.int32)
            ms = []
            for _ in range(6):
                for args in ((o, d, z, z, z), (z, z, o, d, np.ones(k, np.int32))):
                    st = g.apply_batch(*args, stats=True)
                    assert st.n_del_applied + st.n_add_applied == k
                    ms.append(st.ms_phase[sp.PHASES.index("merge")])
            best[k] = min(ms)
        d = g.get_dist()
        assert d[0] == 0 and (d[1:] == 1).all()
        got = g.export_csr()
        for x, y in zip(got, (ro, col, np.ones(n - 1, np.int32))):
            np.testing.assert_array_equal(x, y)
    assert best[1] < 3 * best[700] + 0.02, best
