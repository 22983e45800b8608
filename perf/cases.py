"""What libsp's users run, as cases that can be timed and compared.

The cases are the calls of `sp.Graph` over the sizes that this repository's
workloads, tests and benchmark use: update batches on resident graphs (from a
64-update batch on a thousand vertices to a million updates on 67 million
edges, host and device inputs, every push schedule), from-scratch solves,
loading and saving a graph, dynamic and static PageRank, and the dynamic and
static triangle count.

A batch case applies a batch and then the batch that takes it back (what was
inserted leaves, what was deleted returns with its old weight), as a window
over an edge stream does, so that a pass leaves the edge set as it found it.
Graphs and batches are made on the GPU with torch from the seed alone.
Parents are left out of the outputs: where two tight edges tie, any of them
is a valid parent, and which one wins is not fixed.
"""
import math

import numpy as np
import torch

from paper_2507_11094_gb300 import sp

DAMPING, BETA, MAX_ITER = 0.85, 1e-6, 100    # the repository's PageRank settings
RMAT = (0.57, 0.19, 0.19)                    # quadrants a, b, c of R-MAT


def listed():
    return [
        # the smallest call: 64 updates from plain numpy arrays; launches,
        # synchronisation and host work are all there is
        dict(name="er1k-64", do="batch", graph="er", n=1024, m=8192, updates=64, io="numpy",
             delta=0, pool=0, local=4096),
        # an odd-sized uniform random graph and batches whose deletion and
        # insertion counts differ from call to call, as a live stream's do
        dict(name="er100k-1001", do="batch", graph="er", n=100003, m=1000003, updates=1001,
             io="device", delta=0, pool=0, local=4096),
        # the benchmark's workload, end to end: 1% of R-MAT 20 through
        # page-locked host arrays, every distance back in one
        dict(name="rmat20-1pct", do="batch", graph="rmat", scale=20, factor=16, updates=167772,
             io="pinned", delta=800, pool=0, local=1024),
        # the serving mix's largest request: a million updates on R-MAT 22
        dict(name="rmat22-1M", do="batch", graph="rmat", scale=22, factor=16, updates=1000000,
             io="device", delta=800, pool=0, local=4096),
        # a road-like grid of odd sides, 1%, with the block-local schedule
        # that the tuner picks for grids
        dict(name="grid2047x1531-1pct", do="batch", graph="grid", rows=2047, cols=1531,
             updates=125233, io="device", delta=32000, pool=64, local=0),
        # the batched form: many graphs in one handle, one union batch
        dict(name="batched32", do="batch", graph="batched", count=32, lo=12, hi=16, factor=16,
             frac=0.0275, io="device", delta=800, pool=0, local=4096),
        # the from-scratch solve that every graph starts with
        dict(name="solve-rmat20", do="solve", graph="rmat", scale=20, factor=16, delta=800,
             pool=0, local=1024),
        # a graph comes in (a server's reload): build both stores, solve, and
        # export the edge set again (its checkpoint)
        dict(name="load-rmat20", do="load", graph="rmat", scale=20, factor=16, delta=0, pool=0,
             local=4096),
        # static PageRank, and one dynamic PageRank batch of 1%
        dict(name="pr-rmat20", do="pr", graph="rmat", scale=20, factor=16),
        dict(name="pr-rmat18-1pct", do="pr_batch", graph="rmat", scale=18, factor=16,
             updates=41943),
        # static triangle count, and a batch of 1% of the pairs
        dict(name="tc-rmat18", do="tc", graph="sym-rmat", scale=18, factor=8),
        dict(name="tc-rmat18-1pct", do="tc_batch", graph="sym-rmat", scale=18, factor=8,
             pairs=20971),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same ranges."""
    do = rng.choice(("batch", "batch", "batch", "batch", "solve", "load", "pr", "pr_batch", "tc",
                     "tc_batch"))
    frac = math.exp(rng.uniform(math.log(0.0005), math.log(0.05)))
    if do in ("tc", "tc_batch"):
        if rng.random() < 0.5:
            scale, factor = rng.randint(12, 17), rng.randint(4, 8)
            c = dict(graph="sym-rmat", scale=scale, factor=factor)
            m = factor << scale
        else:
            n = _log(rng, 1000, 400000)
            m = n * rng.randint(3, 16)
            c = dict(graph="sym-er", n=n, m=m)
        if do == "tc_batch":
            c["pairs"] = max(2, int(frac * m))
        return dict(c, do=do)
    # (a plain grid has no random structure, so static PageRank draws none)
    kind = rng.choice(("er", "rmat", "rmat", "grid", "batched") if do == "batch" else
                      ("er", "rmat") if do == "pr" else ("er", "rmat", "grid"))
    mean = 50
    if kind == "er":
        n = _log(rng, 1000, 1000000)
        m = n * rng.randint(4, 16) + rng.randint(0, 99)
        c = dict(graph="er", n=n, m=m)
    elif kind == "rmat":
        scale, factor = rng.randint(10, 20), rng.randint(8, 16)
        c = dict(graph="rmat", scale=scale, factor=factor)
        m = factor << scale
    elif kind == "grid":
        rows, cols = _log(rng, 30, 1500), _log(rng, 30, 1500)
        c = dict(graph="grid", rows=rows, cols=cols)
        m = 4 * rows * cols - 2 * (rows + cols)
        mean = 500
    else:
        lo = rng.randint(10, 13)
        c = dict(graph="batched", count=rng.randint(2, 32), lo=lo, hi=lo + rng.randint(0, 3),
                 factor=rng.randint(8, 16), frac=round(frac, 5))
    if do in ("batch", "pr_batch") and kind != "batched":
        c["updates"] = max(2, int(frac * m))
    if do == "batch":
        c["io"] = rng.choice(("numpy", "pinned", "device", "device"))
    if do in ("batch", "solve", "load"):
        if kind == "grid":
            c.update(delta=64 * mean, pool=64, local=0)
        else:
            c.update(delta=rng.choice((0, 16 * mean)), pool=0, local=rng.choice((1024, 4096)))
    return dict(c, do=do)


# --------------------------------------------------------------------------
# inputs, on the GPU
# --------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 12345)
    return g


def _randint(g, lo, hi, k):
    return torch.randint(lo, hi, (k,), generator=g, device="cuda", dtype=torch.int64)


class _Part:
    """One graph of a handle: vertices [base, base + n), its edge keys
    u * N + v (N = all vertices of the handle) and how new pairs are drawn."""

    def __init__(self, base, n, keys, pairs):
        self.base, self.n, self.keys, self.pairs = base, n, keys, pairs


def _fresh(keys, m, n_all, g, pairs, want, avoid=None):
    """`want` distinct keys of drawn pairs u != v that are not in `keys`."""
    got = torch.empty(0, dtype=torch.int64, device="cuda")
    for _ in range(64):
        if got.numel() >= want:
            break
        u, v = pairs(int((want - got.numel()) * 1.4) + 256)
        c = (u * n_all + v)[u != v]
        if keys is not None and keys.numel():
            at = torch.searchsorted(keys, c).clamp_(max=keys.numel() - 1)
            c = c[keys[at] != c]
        got = torch.unique(torch.cat([got, c]))
    if got.numel() > want:
        got = got[torch.randperm(got.numel(), generator=g, device="cuda")[:want]]
    return got


def _rmat_pairs(g, scale, perm):
    a, b, c = RMAT

    def pairs(k):
        u = torch.zeros(k, dtype=torch.int64, device="cuda")
        v = torch.zeros_like(u)
        for _ in range(scale):
            r = torch.rand(k, generator=g, device="cuda")
            u.mul_(2).add_(r >= a + b)
            v.mul_(2).add_(((r >= a) & (r < a + b)) | (r >= a + b + c))
        return perm[u], perm[v]
    return pairs


def _rmat_part(g, scale, factor, base, n_all):
    n = 1 << scale
    inner = _rmat_pairs(g, scale, torch.randperm(n, generator=g, device="cuda") + base)
    keys = torch.sort(_fresh(None, 0, n_all, g, inner, min(factor * n, n * (n - 1) // 2)))[0]
    return _Part(base, n, keys, inner)


def _er_part(g, n, m):
    def pairs(k):
        return _randint(g, 0, n, k), _randint(g, 0, n, k)
    return _Part(0, n, torch.sort(_fresh(None, 0, n, g, pairs, min(m, n * (n - 1) // 2)))[0],
                 pairs)


def _grid_part(g, rows, cols):
    n = rows * cols
    v = torch.arange(n, device="cuda")
    i, j = v // cols, v % cols
    ks = []
    for di, dj in ((0, 1), (0, -1), (1, 0), (-1, 0)):
        ok = (i + di >= 0) & (i + di < rows) & (j + dj >= 0) & (j + dj < cols)
        ks.append(v[ok] * n + (v + di * cols + dj)[ok])

    def pairs(k):   # a vertex and one of its 5 x 5 neighbourhood: the diameter stays high
        u = _randint(g, 0, n, k)
        a = (u // cols + _randint(g, -2, 3, k)).clamp_(0, rows - 1)
        b = (u % cols + _randint(g, -2, 3, k)).clamp_(0, cols - 1)
        return u, a * cols + b
    return _Part(0, n, torch.sort(torch.cat(ks))[0], pairs)


def _parts(case, g):
    """The case's graph: all vertices, its parts, and the largest weight."""
    kind = case["graph"]
    if kind in ("er", "sym-er"):
        return case["n"], [_er_part(g, case["n"], case["m"])], 100
    if kind in ("rmat", "sym-rmat"):
        n = 1 << case["scale"]
        return n, [_rmat_part(g, case["scale"], case["factor"], 0, n)], 100
    if kind == "grid":
        return case["rows"] * case["cols"], [_grid_part(g, case["rows"], case["cols"])], 1000
    scales = _scales(case)
    n_all, base, parts = sum(1 << s for s in scales), 0, []
    for s in scales:
        parts.append(_rmat_part(g, s, case["factor"], base, n_all))
        base += 1 << s
    return n_all, parts, 100


def _scales(case):
    return [case["lo"] + i % (case["hi"] - case["lo"] + 1) for i in range(case["count"])]


def _i32(x):
    return x.to(torch.int32).contiguous()


class _Inputs:
    """A case's graph as a CSR, its sources, and a batch with its way back."""

    def __init__(self, case, seed):
        g = _gen(seed)
        n, parts, wmax = _parts(case, g)
        sym = case["graph"].startswith("sym-")
        if sym:   # every pair once, then in both directions with one weight
            p = parts[0]
            u, v = p.keys // n, p.keys % n
            pairs = torch.unique(torch.minimum(u, v) * n + torch.maximum(u, v))
            pw = _randint(g, 1, wmax + 1, pairs.numel())
            keys, w = _both(pairs, pw, n)
        else:
            keys = torch.cat([p.keys for p in parts])
            w = _randint(g, 1, wmax + 1, keys.numel())
        u = keys // n
        self.n, self.m = n, int(keys.numel())
        self.row_off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        self.row_off[1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
        self.col, self.w = _i32(keys % n), _i32(w)
        deg = self.row_off[1:] - self.row_off[:-1]
        self.sources = [0 if case["graph"] == "grid" else
                        p.base + int(torch.argmax(deg[p.base:p.base + p.n])) for p in parts]
        self.there = self.back = None
        if case["do"] == "tc_batch":
            k = min(case["pairs"], pairs.numel() // 2)
            at = torch.randperm(pairs.numel(), generator=g, device="cuda")[:k]

            def new(c):
                a, b = parts[0].pairs(c)
                return torch.minimum(a, b), torch.maximum(a, b)
            add = _fresh(pairs, 0, n, g, new, k)
            aw = _randint(g, 1, wmax + 1, add.numel())
            d, dw = _both(pairs[at], pw[at], n)
            a, aw = _both(add, aw, n)
        elif case["do"] in ("batch", "pr_batch"):
            ds, dws, adds, base = [], [], [], 0
            for p, (nd, na) in zip(parts, _counts(case, parts)):
                at = torch.randperm(p.keys.numel(), generator=g, device="cuda")[:nd]
                ds.append(p.keys[at])
                dws.append(w[base + at])
                adds.append(_fresh(p.keys, 0, n, g, p.pairs, na))
                base += p.keys.numel()
            d, dw, a = torch.cat(ds), torch.cat(dws), torch.cat(adds)
            aw = _randint(g, 1, wmax + 1, a.numel())
        else:
            return
        d32, a32 = (_i32(d // n), _i32(d % n)), (_i32(a // n), _i32(a % n))
        self.there = (*d32, *a32, _i32(aw))
        self.back = (*a32, *d32, _i32(dw))


def _both(pairs, w, n):
    u, v = pairs // n, pairs % n
    keys, at = torch.sort(torch.cat([pairs, v * n + u]))
    return keys, torch.cat([w, w])[at]


def _counts(case, parts):
    if case["graph"] == "batched":
        t = [max(2, int(p.keys.numel() * case["frac"] * (0.2 + 1.6 * i / max(1, len(parts) - 1))))
             for i, p in enumerate(parts)]
    else:
        t = [case["updates"]]
    return [(k // 2, k - k // 2) for k in t]


# --------------------------------------------------------------------------
# the calls
# --------------------------------------------------------------------------

class _State:
    pass


def _graph(x, stream):
    return sp.Graph(x.n, x.row_off, x.col, x.w, stream=stream)


def _schedule(g, case):
    g.set_delta(case["delta"])
    g.set_schedule(8, case["pool"])
    g.set_local_rounds(case["local"])


def _host(t, pinned):
    if not pinned:
        return t.cpu().numpy()
    p = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    p.copy_(t)
    return p.numpy()


def prepare(case, seed):
    s = _State()
    s.case, s.do = case, case["do"]
    x = _Inputs(case, seed)
    s.stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    if s.do == "load":
        s.x = x
        s.row_off, s.col, s.w = (torch.empty_like(t) for t in (x.row_off, x.col, x.w))
        s.dist = torch.empty(x.n, dtype=torch.int32, device="cuda")
        return s
    s.g = _graph(x, s.stream)
    if s.do in ("batch", "solve"):
        _schedule(s.g, case)
        s.source = x.sources[0]
        s.dist = [torch.empty(x.n, dtype=torch.int32, device="cuda") for _ in range(2)]
    if s.do == "batch":
        if len(x.sources) > 1:
            s.g.sssp_init_multi(np.asarray(x.sources, dtype=np.int32))
        else:
            s.g.sssp_init(s.source)
        s.there, s.back = x.there, x.back
        if case["io"] != "device":
            pinned = case["io"] == "pinned"
            s.there, s.back = ([_host(t, pinned) for t in b] for b in (s.there, s.back))
            s.dist = [_host(d, pinned) for d in s.dist]
    elif s.do == "pr_batch":
        s.g.pr_init(DAMPING, BETA, MAX_ITER)
        s.there, s.back = x.there, x.back
    elif s.do == "tc_batch":
        s.g.tc_init()
        s.there, s.back = x.there, x.back
    torch.cuda.synchronize()
    return s


def run(s):
    if s.do == "batch":
        s.g.apply_batch_get(*s.there, dist=s.dist[0])
        s.g.apply_batch_get(*s.back, dist=s.dist[1])
        return {"there": s.dist[0], "back": s.dist[1], "edges": s.g.m}
    if s.do == "solve":
        s.g.sssp_init(s.source)
        s.g.get_dist(out=(s.dist[0], None))
        return s.dist[0]
    if s.do == "load":
        with _graph(s.x, s.stream) as g:
            _schedule(g, s.case)
            g.sssp_init(s.x.sources[0])
            g.get_dist(out=(s.dist, None))
            g.export_csr_device(s.row_off, s.col, s.w)
        return {"dist": s.dist, "row_off": s.row_off, "col": s.col, "w": s.w}
    if s.do == "pr":
        s.g.pr_init(DAMPING, BETA, MAX_ITER)
        return s.g.pr_get()
    if s.do == "pr_batch":
        s.g.pr_apply_batch(*s.there)
        there = s.g.pr_get()
        s.g.pr_apply_batch(*s.back)
        return {"there": there, "back": s.g.pr_get()}
    if s.do == "tc":
        return s.g.tc_init()
    return {"there": s.g.tc_apply_batch(*s.there), "back": s.g.tc_apply_batch(*s.back)}


def _sizes(case):
    """Vertices and edges of a case's graph (about)."""
    kind = case["graph"]
    if kind in ("er", "sym-er"):
        n, m = case["n"], case["m"]
    elif kind in ("rmat", "sym-rmat"):
        n = 1 << case["scale"]
        m = case["factor"] * n
    elif kind == "grid":
        n = case["rows"] * case["cols"]
        m = 4 * n - 2 * (case["rows"] + case["cols"])
    else:
        n = sum(1 << s for s in _scales(case))
        m = case["factor"] * n
    return n, 2 * m if kind.startswith("sym-") else m


def work(case):
    """The bytes a pass cannot do without: every input array and every edge
    that decides the answer read once, every output and changed edge (8 bytes
    in each of the two stores) written once.  A floating operation is one add
    per pulled in-edge and Jacobi step; PageRank takes some 20 steps to reach
    BETA, each of which has to read the ranks of the one before."""
    n, m = _sizes(case)
    do = case["do"]
    if do == "batch":
        k = case["updates"] if "updates" in case else case["frac"] * m
        return {"bytes": 2 * (k * 10 + k * 16 + 4 * n), "flops": 0}
    if do == "solve":
        return {"bytes": 8 * m + 8 * n + 4 * n, "flops": 0}
    if do == "load":   # in, two stores, a solve, out
        return {"bytes": 8 * m + 8 * n + 16 * m + 8 * m + 4 * n + 8 * m + 8 * n, "flops": 0}
    if do == "pr":
        return {"bytes": 20 * (4 * m + 8 * n) + 4 * n, "flops": 20 * m}
    if do == "pr_batch":   # two batches of two phases each
        return {"bytes": 4 * 10 * (4 * m + 8 * n) + 8 * n, "flops": 4 * 10 * m}
    if do == "tc":
        return {"bytes": 4 * m + 8 * n, "flops": 0}
    return {"bytes": 2 * (4 * case["pairs"] * 10 + 4 * case["pairs"] * 16), "flops": 0}


# --------------------------------------------------------------------------
# the same in 64 bits
# --------------------------------------------------------------------------

def _jacobi(u, v, pr, sel, n):
    """Jacobi steps over the vertices `sel` (a mask) until they change by at
    most BETA in all, or MAX_ITER of them."""
    damping = float(np.float32(DAMPING))    # the entry point takes a 32-bit float
    outdeg = torch.bincount(u, minlength=n).double()
    base = (1.0 - damping) / n
    keep = sel[v]
    eu, ev = u[keep], v[keep]
    for _ in range(MAX_ITER):
        term = torch.where(outdeg > 0, pr / outdeg.clamp(min=1.0), torch.zeros_like(pr))
        acc = torch.zeros_like(pr).index_add_(0, ev, term[eu])
        new = torch.where(sel, base + damping * acc, pr)
        diff = float((new - pr).abs().sum())
        pr = new
        if diff <= BETA:
            break
    return pr


def _reach(u, v, start, n):
    """The vertices reachable from `start` along edges, those among them."""
    hit = torch.zeros(n, dtype=torch.bool, device="cuda")
    hit[start] = True
    while True:
        nxt = hit.clone()
        nxt[v[hit[u]]] = True
        if bool((nxt == hit).all()):
            return hit
        hit = nxt


def exact(case, seed):
    if case["do"] not in ("pr", "pr_batch"):
        return None    # distances, edges and counts are whole numbers
    x = _Inputs(case, seed)
    n = x.n
    u = torch.repeat_interleave(torch.arange(n, device="cuda"), x.row_off[1:] - x.row_off[:-1])
    keys = u * n + x.col.long()
    everything = torch.ones(n, dtype=torch.bool, device="cuda")
    pr = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    pr = _jacobi(keys // n, keys % n, pr, everything, n)
    if case["do"] == "pr":
        return pr.cpu().numpy()
    out = {}
    for name, (ds, dd, as_, ad, _) in (("there", x.there), ("back", x.back)):
        # deletions flag on the graph before them, insertions on the one
        # before the insertions; each phase's steps run on the updated graph
        sel = _reach(keys // n, keys % n, dd.long(), n)
        keys = keys[~torch.isin(keys, ds.long() * n + dd.long())]
        pr = _jacobi(keys // n, keys % n, pr, sel, n)
        sel = _reach(keys // n, keys % n, ad.long(), n)
        keys = torch.sort(torch.cat([keys, as_.long() * n + ad.long()]))[0]
        pr = _jacobi(keys // n, keys % n, pr, sel, n)
        out[name] = pr.cpu().numpy()
    return out
