"""GPU tests of the algorithmic bytes that a call reports: they follow the passes
and paths that its kernels took."""
import numpy as np
import pytest

from paper_2507_11094_gb300 import sp
from paper_2507_11094_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
PH = {p: i for i, p in enumerate(sp.PHASES)}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2507_11094_gb300 import build
    build.build()
    sp.load()


def insertions(n, k, seed):
    rng = np.random.default_rng(seed)
    key = rng.choice(n * n, size=k, replace=False)
    i32 = lambda x: np.ascontiguousarray(x, np.int32)
    z = np.zeros(0, np.int32)
    return wl.Batch(z, z, i32(key // n), i32(key % n), i32(rng.integers(1, 101, k)))


# id bits b, items and the passes over them: 2 b key bits in two halves of the
# grid (one more in one block, up to 4,096 items) in digits of nine bits, or of
# ten where these are fewer; none where one block plans the batch
@pytest.mark.parametrize("n,k,passes", [
    (600, 1024, 0), (600, 1025, 3), (600, 2048, 3), (600, 4000, 2), (500, 4000, 2),
    (1100, 4000, 3), (5000, 1500, 3), (5000, 4000, 3), (300000, 1500, 4), (300000, 4000, 4)])
def test_sort_bytes(n, k, passes):
    ro, col, w = wl.er_digraph(n, 2000, 1, 100, seed=n)
    with sp.Graph(n, ro, col, w) as g:
        g.sssp_init(0)
        st = g.apply(insertions(n, k, n), stats=True)
    rows = st.rows_touched
    if passes == 0:
        assert st.alg_bytes[PH["sort"]] == 10 * k
        assert st.alg_bytes[PH["count"]] == 51 * 2 * k + 16 * rows
    else:
        assert st.alg_bytes[PH["sort"]] == 20 * k + 2 * k * (12 + 24 * passes + 34)
        assert st.alg_bytes[PH["count"]] == 37 * 2 * k + 16 * rows


def test_rank_bytes():
    n, m = 3000, 20000
    ro, col, w = wl.er_digraph(n, m, 1, 100, seed=1)
    with sp.Graph(n, ro, col, w) as g:
        st = g.pr_init(0.85, 1e-6, 100, stats=True)
        assert st.alg_bytes[PH["pull"]] == 8 * st.relaxed_edges + 24 * n * st.rounds_push
        st = g.pr_apply(insertions(n, 700, 2), stats=True)   # one phase
        assert st.alg_bytes[PH["pull"]] == (8 * st.relaxed_edges +
                                            24 * st.affected * st.rounds_push)


def test_the_count_phase_of_a_triangle_batch():
    # phases are those of an update batch: the plan of a small one (1,000 updates:
    # searches, sort and count in one block) is of the count phase, after a sort
    # phase in which only the control block is reset
    import torch
    W = wl.sym_er(65536, 600000, 250, 3)
    sort, count = [], []
    with sp.Graph(W.n, W.row_off, W.col, W.w) as g:
        g.tc_init()
        for k in range(6):
            b = W.batch(k)
            assert b.size <= 1024
            dev = [torch.from_numpy(x).cuda() for x in
                   (b.del_src, b.del_dst, b.add_src, b.add_dst, b.add_w)]
            _, st = g.tc_apply_batch(*dev, stats=True)
            sort.append(st.ms_phase[PH["sort"]])
            count.append(st.ms_phase[PH["count"]])
    assert min(sort) < 0.5 * min(count), (sort, count)
