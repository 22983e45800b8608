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
