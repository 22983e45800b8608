"""GPU tests of the searches of a batch's updates in their old rows, over rows
that an interpolating search finds hard: clustered cols, cols that double, and
hits and misses at and beyond a row's ends, in both stores.  A batch that one
block plans always interpolates; the grid's searches do from 1 GiB a store on
(reached here by rows with slack)."""
import numpy as np
import pytest

import oracle
from paper_2507_11094_gb300 import sp
from paper_2507_11094_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
N = 200000


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2507_11094_gb300 import build
    build.build()
    oracle.build()
    sp.load()


def hard_rows():
    """Col sets by row: lengths around four sectors of four entries (up to which
    a row's ends are not read first), and longer."""
    a = np.arange
    rows = [a(k) * 3 + 50 for k in (1, 2, 3, 4, 5, 15, 16, 17, 18, 33)]
    rows += [np.r_[a(1000, 6000), N - 1],                        # a run and one far col
             np.r_[0, a(N - 7001, N - 1)],
             np.r_[a(500), a(N // 2, N // 2 + 500), a(N - 500, N)],
             np.unique((1.01 ** a(1100)).astype(np.int64)),       # ever wider apart
             N - 1 - np.unique((1.5 ** a(29)).astype(np.int64)),
             np.r_[0, 1, 2, a(5000) + 100000, N - 2, N - 1],
             a(0, N, 2)]
    return [np.unique(r[(r >= 0) & (r < N)]) for r in rows]


def graph(fill):
    """The hard rows as rows of the forward store and as rows of the reverse one,
    and `fill` random edges among other vertices."""
    rows = hard_rows()
    src = 1000 + 7 * np.arange(len(rows))
    dst = 1003 + 7 * np.arange(len(rows))
    keys = [s * N + r for s, r in zip(src, rows)] + [r * N + d for d, r in zip(dst, rows)]
    rng = np.random.default_rng(fill)
    keys.append(rng.integers(2000, N, fill) * N + rng.integers(2000, N, fill))
    keys = np.unique(np.concatenate(keys))
    ro = np.zeros(N + 1, np.int64)
    np.cumsum(np.bincount(keys // N, minlength=N), out=ro[1:])
    return keys, ro, (keys % N).astype(np.int32), rng.integers(1, 101, keys.size).astype(np.int32)


def updates(keys, k, rng):
    """k updates of the hard rows: their ends, what lies beyond and between."""
    rows = hard_rows()
    every = []
    for i, r in enumerate(rows):
        at = np.unique(np.r_[0, 1, 2, 3, 4, r.size - 2, r.size - 1,
                             rng.integers(0, r.size, 1 + k // (4 * len(rows)))])
        c = r[at[(at >= 0) & (at < r.size)]]
        c = np.unique(np.r_[c, c - 1, c + 1, 0, N - 1, rng.integers(0, N, 8)])
        c = c[(c >= 0) & (c < N)]
        every += [(1000 + 7 * i) * N + c, c * N + (1003 + 7 * i)]
    every = rng.permutation(np.unique(np.concatenate(every)))[:k]
    present = np.isin(every, keys)
    goes = np.where(present, rng.random(every.size) < 0.8, rng.random(every.size) < 0.2)
    gone = every[goes]                                           # some are absent
    new = every[~present | (rng.random(every.size) < 0.3)]       # some are present, or go and come
    i32 = lambda x: np.ascontiguousarray(x, np.int32)
    return wl.Batch(i32(gone // N), i32(gone % N), i32(new // N), i32(new % N),
                    i32(rng.integers(1, 101, new.size)))


# one block's plan, and the grid's halving and interpolating searches
@pytest.mark.parametrize("fill,slack,k", [(1000, 0.25, 600), (1000, 0.25, 3000),
                                          (3300000, 16.0, 3000), (3300000, 16.0, 600)])
def test_searches_in_hard_rows(fill, slack, k):
    keys, ro, col, w = graph(fill)
    ref = oracle.OracleGraph(N, ro, col, w)
    rng = np.random.default_rng(k)
    with sp.Graph(N, ro, col, w, slack=slack) as g:
        big = max(g.info().cap_fwd, g.info().cap_rev) * 8 >= 1 << 30
        assert big == (slack == 16.0)
        g.sssp_init(1000)
        for _ in range(2):
            rro, rcol, _ = ref.csr()
            b = updates(wl.csr_keys(N, rro, rcol), k, rng)
            assert (b.size <= 1024) == (k == 600)
            want = ref.apply(b)
            st = g.apply(b, stats=True)
            assert (st.n_del_applied, st.n_del_absent, st.n_add_applied, st.n_add_present) == want
            assert min(want) > 0
            for x, y in zip(g.export_csr(), ref.csr()):
                np.testing.assert_array_equal(x, y)
        ro, col, w = ref.csr()
        u = np.repeat(np.arange(N), np.diff(ro))
        order = np.lexsort((u, col))
        rro, rcol, rw = g.export_csr(reverse=True)
        np.testing.assert_array_equal(np.diff(rro), np.bincount(col, minlength=N))
        np.testing.assert_array_equal(rcol, u[order])
        np.testing.assert_array_equal(rw, w[order])
