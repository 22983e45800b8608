"""GPU tests of host arrays handed to a batch: they are read in stream order
where work on the graph's stream may still be writing them."""
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


def batch(ref, n, k, rng):
    """k updates: half present edges go, half new ones come."""
    ro, col, _ = ref.csr()
    keys = wl.csr_keys(n, ro, col)
    gone = rng.choice(keys, size=k // 2, replace=False)
    new = rng.choice(np.setdiff1d(rng.integers(0, n * n, 4 * k), keys), size=k - k // 2,
                     replace=False)
    i32 = lambda x: np.ascontiguousarray(x, np.int32)
    return [i32(gone // n), i32(gone % n), i32(new // n), i32(new % n),
            i32(rng.integers(1, 101, new.size))]


# page-locked arrays (by position) whose contents come from a copy that is
# queued on the graph's stream behind other work when the call is made; the
# others are ordinary memory.  Small batches, the largest small one, and more
@pytest.mark.parametrize("k", [6, 1024, 1026])
@pytest.mark.parametrize("pinned", [(0, 1, 2, 3, 4), (0, 1, 2, 3), (0, 1), (2, 3, 4), (4,), ()])
def test_arrays_that_queued_work_still_fills(k, pinned):
    import torch
    n = 3000
    ro, col, w = wl.er_digraph(n, 20000, 1, 100, seed=3)
    ref = oracle.OracleGraph(n, ro, col, w)
    rng = np.random.default_rng(k)
    st = torch.cuda.Stream()
    with sp.Graph(n, ro, col, w, stream=st) as g:
        g.sssp_init(0)
        old = batch(ref, n, k, rng)            # valid ids, but not this call's
        for _ in range(3):                     # the third call replays a cached graph
            b = batch(ref, n, k, rng)
            args, keep = [], []
            for q in range(5):
                if q not in pinned:
                    args.append(b[q])
                    continue
                host = torch.empty(b[q].size, dtype=torch.int32, pin_memory=True)
                host.copy_(torch.from_numpy(old[q]))
                keep.append((host, torch.from_numpy(b[q]).cuda()))
                args.append(host.numpy())
            torch.cuda.synchronize()
            with torch.cuda.stream(st):
                torch.cuda._sleep(20_000_000)
                for host, dev in keep:
                    host.copy_(dev, non_blocking=True)
            dist, parent = np.full(n, -7, np.int32), np.full(n, -7, np.int32)
            g.apply_batch_get(*args, dist=dist, parent=parent)
            ref.apply(wl.Batch(*b))
            np.testing.assert_array_equal(dist, ref.dijkstra(0))
            for x, y in zip(g.export_csr(), ref.csr()):
                np.testing.assert_array_equal(x, y)
            old = b


# page-locked arrays of a small batch that another thread keeps changing, to ids
# out of range too, while the call runs: they are read once, so what was checked
# is what is applied, or nothing is (a mix of two batches at worst)
@pytest.mark.parametrize("k", [6, 1024])
def test_arrays_that_change_during_the_call(k):
    import threading
    import torch
    n = 3000
    ro, col, w = wl.er_digraph(n, 20000, 1, 100, seed=3)
    rng = np.random.default_rng(k)
    ref = oracle.OracleGraph(n, ro, col, w)
    two = [batch(ref, n, k, rng) for _ in range(2)]
    pins = [torch.empty(a.size, dtype=torch.int32, pin_memory=True).numpy() for a in two[0]]
    stop = threading.Event()

    def change():
        i = 0
        while not stop.is_set():
            i += 1
            for p, a in zip(pins, two[i % 2]):
                p[:] = a
            if i % 3 == 0:
                pins[1][::2] = 0x7FFFFFF0
                pins[3][1::2] = -5
    with sp.Graph(n, ro, col, w, stream=torch.cuda.Stream()) as g:
        g.sssp_init(0)
        for p, a in zip(pins, two[0]):
            p[:] = a
        t = threading.Thread(target=change)
        t.start()
        codes = set()
        for _ in range(300):
            codes.add(g.apply_batch(*pins, raise_on_error=False)[0])
        stop.set()
        t.join()
        assert codes <= {sp.SP_OK, sp.SP_EINVAL}
        ref = oracle.OracleGraph(n, *g.export_csr())
        assert g.m == ref.csr()[1].size
        np.testing.assert_array_equal(g.get_dist(), ref.dijkstra(0))
