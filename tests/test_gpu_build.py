"""GPU tests of building a graph's stores from a CSR and exporting them: the
forward and the reverse store against numpy, over rows, gaps and edge counts at
the bounds of what a warp walks (1,024 edges, windows of 32 rows) and of the
edge sort's tiles (4,096 pairs, digits of at most eight bits)."""
import numpy as np
import pytest

from paper_2507_11094_gb300 import sp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2507_11094_gb300 import build
    build.build()
    sp.load()


def edges(n, m, kind, seed):
    """Distinct (u, v) keys u * n + v, sorted."""
    rng = np.random.default_rng(seed)
    if kind == "uniform":
        k = rng.integers(0, n * n, size=3 * m + 64)
    elif kind == "hub":      # half of the edges leave one vertex, half enter another
        half = m // 2
        v = rng.permutation(n)[:half]
        u = rng.permutation(n)[:m - half]
        k = np.concatenate([(n // 2) * n + v, u * n + n // 3])
    elif kind == "gaps":     # edges in a few far rows only, the first and last among them
        rows = np.unique(np.concatenate([[0, n - 1], rng.integers(0, n, size=max(1, m // 40))]))
        k = rng.choice(rows, size=3 * m + 64) * n + rng.integers(0, n, size=3 * m + 64)
    k = np.unique(k)
    if k.size > m:
        k = np.sort(rng.choice(k, size=m, replace=False))
    return k


def csr(n, keys, w, reverse=False):
    u, v = keys // n, keys % n
    if reverse:
        order = np.lexsort((u, v))
        u, v, w = v[order], u[order], w[order]
    ro = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(u, minlength=n), out=ro[1:])
    return ro, v.astype(np.int32), w.astype(np.int32)


@pytest.mark.parametrize("n,m,kind", [
    (1, 0, "uniform"), (2, 1, "uniform"), (31, 200, "uniform"), (100, 1023, "uniform"),
    (100, 1024, "uniform"), (100, 1025, "uniform"), (255, 4095, "uniform"),
    (256, 4096, "uniform"), (257, 4097, "uniform"), (5000, 8193, "hub"), (40000, 60000, "hub"),
    (200000, 4000, "gaps"), (3000000, 97, "gaps"), (65537, 300000, "uniform"),
    (300001, 1000003, "uniform")])
def test_stores_of_a_csr(n, m, kind):
    keys = edges(n, m, kind, seed=n + m)
    w = np.random.default_rng(1).integers(1, sp.SP_WMAX + 1, size=keys.size)
    ro, col, ww = csr(n, keys, w)
    rng = np.random.default_rng(2)
    mixed = np.argsort(rng.random(col.size) + np.repeat(np.arange(n), np.diff(ro)))
    for order in (np.arange(col.size), mixed):   # rows in order, and not
        with sp.Graph(n, ro, col[order], ww[order]) as g:
            for rev in (False, True):
                for got, want in zip(g.export_csr(reverse=rev), csr(n, keys, w, rev)):
                    np.testing.assert_array_equal(got, want)
    if keys.size > 1:   # an edge twice, in order and not
        i = int(rng.integers(0, keys.size))
        for k in (np.insert(keys, i, keys[i]), None):
            if k is None:
                r = int(np.argmax(np.diff(ro)))
                if ro[r + 1] - ro[r] < 3:
                    continue
                bad = col.copy()
                bad[ro[r + 1] - 1] = bad[ro[r]]
                args = (ro, bad, ww)
            else:
                args = csr(n, k, np.insert(w, i, 1))
            with pytest.raises(sp.SpError) as e:
                sp.Graph(n, *args)
            assert e.value.code == sp.SP_EINVAL


# graphs with far fewer edges than vertices, in part or in whole: a warp's window
# of rows gets wider, among dense rows too, at every distance between edges
@pytest.mark.parametrize("n,gaps", [(70000, (1, 2, 15, 16, 17)), (3000001, (31, 33, 255, 256, 511)),
                                    (5000000, (4095, 4096, 8191, 70000)), (4000000, (1, 900, 1))])
def test_stores_of_sparse_rows(n, gaps):
    rng = np.random.default_rng(n)
    rows = []
    at = 0
    for k in range(400):          # runs of rows `gap` apart, dense rows between them
        gap = gaps[k % len(gaps)]
        rows.append(at + gap * np.arange(60))
        at = int(rows[-1][-1]) + gap
        if k % 7 == 3:
            rows.append(np.full(int(rng.integers(1, 1500)), at))
            at += 1
        if at >= n - 70 * max(gaps):
            break
    u = np.r_[0, np.concatenate(rows), n - 1]
    key = np.unique(np.minimum(u, n - 1) * n + rng.integers(0, n, u.size))
    w = rng.integers(1, sp.SP_WMAX + 1, size=key.size)
    ro, col, ww = csr(n, key, w)
    with sp.Graph(n, ro, col, ww) as g:
        for rev in (False, True):
            for got, want in zip(g.export_csr(reverse=rev), csr(n, key, w, rev)):
                np.testing.assert_array_equal(got, want)


def test_few_edges_among_many_vertices_are_not_slow():
    # 10,000 edges on 10 M vertices load and export in less time than 10 M edges
    # on as many (warps that walked 32 rows at a time took three times as long)
    import time
    import torch
    n = 10 ** 7
    best = {}
    for m in (10 ** 4, 10 ** 7):
        k = np.unique(np.random.default_rng(m).integers(0, n * n, m))
        ro, col, w = csr(n, k, np.ones(k.size, np.int64))
        d = [torch.from_numpy(x).cuda() for x in (ro, col, w)]
        o = [torch.empty_like(x) for x in d]
        load, export = [], []
        for _ in range(5):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            with sp.Graph(n, *d) as g:
                t1 = time.perf_counter()
                g.export_csr_device(*o)
                t2 = time.perf_counter()
            load.append(t1 - t0)
            export.append(t2 - t1)
        assert all(torch.equal(x, y) for x, y in zip(d, o))
        best[m] = min(load), min(export)
    assert best[10 ** 4][0] < best[10 ** 7][0] and best[10 ** 4][1] < best[10 ** 7][1], best
