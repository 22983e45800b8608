// sp_tc.cu -- dynamic triangle count (paper, appendix listing "Dynamic TC
// coded in StarPlat DSL": staticTC, Decremental, Incremental, DynTC).
//
// The graph is read as undirected: every edge is stored in both directions
// (checked).  staticTC counts every triangle once; the listing sees it at its
// middle vertex by id (u < v < w), the kernels here at its smallest one by
// (degree, id), which is the same number.
// A batch changes the count by the listing's corrections.  For every
// applied update (v1, v2) (each pair appears in both directions) and every
// common neighbour v3 of v1 and v2, the triangle {v1, v2, v3} is seen once
// per updated edge it contains and per direction, so with k of its three
// edges updated it is seen 2k times: the correction is
//     count1 / 2 + count2 / 4 + count3 / 6
// where count_k counts the sightings with k updated edges.  Deletions are
// counted on the graph before the merge (Decremental) and subtracted,
// insertions on the graph after it (Incremental) and added.  The common
// neighbours are found by walking the shorter of the two sorted rows and
// binary-searching the other, which finds the same set as the listing's
// walk over v1's row.
#include <algorithm>

#include "sp_graph.cuh"

namespace sp {

namespace {

constexpr int kThreads = 256;
constexpr u32 kFull = 0xffffffffu;

__device__ __forceinline__ u64 warp_sum64(u64 x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
  return x;
}

__device__ __forceinline__ u32 warp_incl_scan(u32 x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u32 y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// Lane holding the warp-wide element t, given the lanes' inclusive counts
// (t < the total): the number of lanes whose count is at most t.
__device__ __forceinline__ int owner_lane(u32 incl, u32 t) {
  int o = 0;
#pragma unroll
  for (int step = 16; step > 0; step >>= 1)
    if (__shfl_sync(kFull, incl, o + step - 1) <= t) o += step;
  return o;
}

// --- staticTC ---------------------------------------------------------------
//
// Every undirected edge {u, v} is kept once, from the end that is smaller by
// (degree, id), which bounds the lists by sqrt(2 m) whatever the hubs; a
// triangle is then seen once, at its smallest vertex u: v in out(u), w in
// out(u) and w in out(v).  k_tc_orient writes out(v) as plain u32 ids into
// row v's alternate region of the forward store (free between merges, and at
// least as long as the row), so the count needs no memory of its own.  In the
// same pass every row is compared with the same row of the reverse store:
// equal rows everywhere mean that every edge has its reverse, which is the
// symmetry check without a search per edge.  R-MAT 18, edge factor 8: check and
// count 0.54 ms; a warp per vertex v walking its lower neighbours one by one,
// behind a binary search per edge, took 29.3 ms (1.14 ms of it the check):
// the hubs' rows were serial.
constexpr int kOrientRow = 256;      // longer rows are taken by a whole block
constexpr int kOrientGiant = 65536;  // ... and these by the whole grid
constexpr int kOK = 4;               // edges per thread in flight

struct OrientArgs {
  Store fwd, rev;
  u32 *cnt;       // [n] |out(v)|
  u32 *giant;     // rows for k_tc_orient_giant
  Ctl *c;
  int n, rpw;     // rows per warp (1..32)
};

struct OrientEdge {   // one edge of row v, its loads issued apart from their use
  int x, y, dx;
};

__device__ __forceinline__ void orient_load(const OrientArgs &a, long long fs, long long rs, u32 e,
                                            bool on, OrientEdge &g) {
  g.x = on ? __ldg(&a.fwd.adj[fs + e].x) : 0;
  g.y = on ? __ldg(&a.rev.adj[rs + e].x) : 0;
}

// Does v keep the edge to x: is v smaller by (degree, id)?
__device__ __forceinline__ bool orient_keeps(int v, int dv, int x, int dx) {
  return x != v && (dx > dv || (dx == dv && x > v));
}

__global__ void __launch_bounds__(kThreads) k_tc_orient(OrientArgs a) {
  __shared__ u32 s_cnt[kThreads / 32][32];
  __shared__ u32 s_row[kThreads], s_nrow, s_out;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rpb = a.rpw * (kThreads / 32);
  bool bad = false;
  for (long long b0 = (long long)blockIdx.x * rpb; b0 < a.n; b0 += (long long)gridDim.x * rpb) {
    if (threadIdx.x == 0) s_nrow = 0;
    s_cnt[warp][lane] = 0;
    __syncthreads();
    // the warp's rows, one per lane, then their edges spread over the lanes
    const long long r = b0 + (long long)warp * a.rpw + lane;
    const bool mine = lane < a.rpw && r < a.n;
    int deg = 0;
    long long fs = 0, rs = 0, alt = 0;
    if (mine) {
      const RowMeta f = a.fwd.row[r], q = a.rev.row[r];
      deg = f.deg;
      fs = f.start;
      rs = q.start;
      alt = a.fwd.alt[r];
      if (q.deg != f.deg) {
        bad = true;
        deg = 0;     // not symmetric: the count is not kept
      }
    }
    u32 len = (u32)deg;
    if (deg > kOrientGiant) {
      a.giant[atomicAdd(&a.c->tc_ngiant, 1u)] = (u32)r;
      a.cnt[r] = 0;
      len = 0;
    } else if (deg > kOrientRow) {
      s_row[atomicAdd(&s_nrow, 1u)] = (u32)r;
      len = 0;
    }
    const u32 incl = warp_incl_scan(len), total = __shfl_sync(kFull, incl, 31);
    const u32 excl = incl - len;
    for (u32 t0 = 0; t0 < total; t0 += 32 * kOK) {
      OrientEdge g[kOK];
      int o[kOK];
      bool on[kOK];
#pragma unroll
      for (int k = 0; k < kOK; ++k) {
        const u32 t = t0 + 32 * k + lane;
        on[k] = t < total;
        o[k] = owner_lane(incl, on[k] ? t : 0u) & 31;
        const u32 e = t - __shfl_sync(kFull, excl, o[k]);
        orient_load(a, __shfl_sync(kFull, fs, o[k]), __shfl_sync(kFull, rs, o[k]), e, on[k], g[k]);
      }
#pragma unroll
      for (int k = 0; k < kOK; ++k) g[k].dx = on[k] ? __ldg(&a.fwd.row[g[k].x].deg) : 0;
#pragma unroll
      for (int k = 0; k < kOK; ++k) {
        const int dv = __shfl_sync(kFull, deg, o[k]);
        const long long av = __shfl_sync(kFull, alt, o[k]);
        const int v = (int)__shfl_sync(kFull, (u32)r, o[k]);
        if (!on[k]) continue;
        bad |= g[k].x != g[k].y;
        if (orient_keeps(v, dv, g[k].x, g[k].dx))
          ((u32 *)(a.fwd.adj + av))[atomicAdd(&s_cnt[warp][o[k]], 1u)] = (u32)g[k].x;
      }
    }
    __syncwarp();
    if (mine && (u32)deg == len) a.cnt[r] = s_cnt[warp][lane];
    __syncthreads();
    const u32 nrow = s_nrow;
    for (u32 i = 0; i < nrow; ++i) {   // long rows, the whole block on each
      const int v = (int)s_row[i];
      const RowMeta f = a.fwd.row[v];
      const long long rv = a.rev.row[v].start;
      u32 *out = (u32 *)(a.fwd.adj + a.fwd.alt[v]);
      if (threadIdx.x == 0) s_out = 0;
      __syncthreads();
      for (u32 e0 = threadIdx.x; e0 < (u32)f.deg; e0 += kThreads * kOK) {
        OrientEdge g[kOK];
#pragma unroll
        for (int k = 0; k < kOK; ++k)
          orient_load(a, f.start, rv, e0 + k * kThreads, e0 + k * kThreads < (u32)f.deg, g[k]);
#pragma unroll
        for (int k = 0; k < kOK; ++k)
          g[k].dx = e0 + k * kThreads < (u32)f.deg ? __ldg(&a.fwd.row[g[k].x].deg) : 0;
#pragma unroll
        for (int k = 0; k < kOK; ++k) {
          if (e0 + k * kThreads >= (u32)f.deg) continue;
          bad |= g[k].x != g[k].y;
          if (orient_keeps(v, f.deg, g[k].x, g[k].dx)) out[atomicAdd(&s_out, 1u)] = (u32)g[k].x;
        }
      }
      __syncthreads();
      if (threadIdx.x == 0) a.cnt[v] = s_out;
    }
    __syncthreads();
  }
  if (bad) atomicCAS(&a.c->status, 0, SP_EINVAL);
}

// Rows longer than kOrientGiant (at most m / kOrientGiant of them): every
// block takes its share of each.
__global__ void __launch_bounds__(kThreads) k_tc_orient_giant(OrientArgs a) {
  const u32 ng = ld_cg_u32(&a.c->tc_ngiant);
  bool bad = false;
  for (u32 i = 0; i < ng; ++i) {
    const int v = (int)a.giant[i];
    const RowMeta f = a.fwd.row[v];
    const long long rv = a.rev.row[v].start;
    u32 *out = (u32 *)(a.fwd.adj + a.fwd.alt[v]);
    for (long long e = blockIdx.x * (long long)kThreads + threadIdx.x; e < f.deg;
         e += (long long)gridDim.x * kThreads) {
      OrientEdge g;
      orient_load(a, f.start, rv, (u32)e, true, g);
      bad |= g.x != g.y;
      if (orient_keeps(v, f.deg, g.x, __ldg(&a.fwd.row[g.x].deg)))
        out[atomicAdd(a.cnt + v, 1u)] = (u32)g.x;
    }
  }
  if (bad) atomicCAS(&a.c->status, 0, SP_EINVAL);
}

// The lists longer than kWarpList, one block each, in a list of their own
// (those longer than kLongList from its front, the others from its end: a
// block that starts on a long one last would keep the rest of the GPU waiting);
// the shorter ones are taken from the vertices in order, a warp each.
constexpr u32 kWarpList = 32, kLongList = 256;

__global__ void __launch_bounds__(kThreads) k_tc_lists(const u32 *__restrict__ cnt, int n, u32 *big,
                                                       Ctl *c) {
  const int lane = threadIdx.x & 31;
  const long long step = (long long)gridDim.x * kThreads;
  for (long long b = blockIdx.x * (long long)kThreads + (threadIdx.x & ~31); b < n; b += step) {
    const long long v = b + lane;
    const u32 d = v < n ? cnt[v] : 0u;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const bool is = k == 0 ? d > kLongList : d > kWarpList && d <= kLongList;
      const u32 m = __ballot_sync(kFull, is);
      if (!m) continue;
      u32 base = 0;
      if (lane == 0) base = atomicAdd(k == 0 ? &c->tc_nbig : &c->tc_nmid, (u32)__popc(m));
      base = __shfl_sync(kFull, base, 0) + __popc(m & lanemask_lt());
      if (is) big[k == 0 ? base : (u32)n - 1u - base] = (u32)v;
    }
  }
}

constexpr u32 kEmpty = 0xFFFFFFFFu;       // no vertex has this id (n < 2^31)
constexpr u32 kTabMax = 8192;             // slots of a block's table: half of them used at most
constexpr u32 kWarpTab = 1024, kWarpTabBits = 10;   // a warp's, for lists of up to kWarpList
static_assert(kWarpTab * (kThreads / 32) <= kTabMax, "the warps' tables share the block's");
constexpr u32 kWK = 4;                    // probes per lane in flight

__device__ __forceinline__ u32 hash_slot(u32 x, u32 bits) { return (x * 0x9E3779B1u) >> (32 - bits); }

__device__ __forceinline__ void tab_put(u32 *tab, u32 bits, u32 x) {
  const u32 mask = (1u << bits) - 1;
  u32 h = hash_slot(x, bits);
  while (atomicCAS(tab + h, kEmpty, x) != kEmpty) h = (h + 1) & mask;   // ids are distinct
}

// (at most half of the slots are used, so every probe ends)
__device__ __forceinline__ bool tab_has(const u32 *tab, u32 bits, u32 x) {
  const u32 mask = (1u << bits) - 1;
  u32 h = hash_slot(x, bits);
  for (;;) {
    const u32 y = tab[h];
    if (y == x) return true;
    if (y == kEmpty) return false;
    h = (h + 1) & mask;
  }
}

// The elements of the lanes' lists (ptr, len) that are in the table: lists of
// at least 32 elements on average are read one after the other by the whole
// warp, shorter ones are laid end to end over the lanes.
__device__ __forceinline__ u32 count_lists(const u32 *ptr, u32 len, const u32 *tab, u32 bits) {
  const int lane = threadIdx.x & 31;
  const u32 incl = warp_incl_scan(len), total = __shfl_sync(kFull, incl, 31);
  u32 c = 0;
  u32 lists = __ballot_sync(kFull, len > 0);
  if (total >= 32u * __popc(lists)) {
    while (lists) {
      const int o = __ffs(lists) - 1;
      lists &= lists - 1;
      const u32 *p = (const u32 *)__shfl_sync(kFull, (u64)ptr, o);
      const u32 n = __shfl_sync(kFull, len, o);
      for (u32 e = lane; e < n; e += 32 * kWK) {
        u32 x[kWK];
#pragma unroll
        for (u32 k = 0; k < kWK; ++k) x[k] = e + 32 * k < n ? __ldg(p + e + 32 * k) : kEmpty;
#pragma unroll
        for (u32 k = 0; k < kWK; ++k) c += x[k] != kEmpty && tab_has(tab, bits, x[k]);
      }
    }
  } else {
    const u32 excl = incl - len;
    for (u32 t0 = 0; t0 < total; t0 += 32 * kWK) {
      u32 x[kWK];
#pragma unroll
      for (u32 k = 0; k < kWK; ++k) {
        const u32 t = t0 + 32 * k + lane;
        const int o = owner_lane(incl, t < total ? t : 0u) & 31;
        const u32 *p = (const u32 *)__shfl_sync(kFull, (u64)ptr, o);
        const u32 e = t - __shfl_sync(kFull, excl, o);
        x[k] = t < total ? __ldg(p + e) : kEmpty;
      }
#pragma unroll
      for (u32 k = 0; k < kWK; ++k) c += x[k] != kEmpty && tab_has(tab, bits, x[k]);
    }
  }
  return c;
}

// One vertex u at a time: out(u) in a hash table in shared memory, then the
// lists of its members walked coalesced and looked up there.  A list longer
// than half a block's table is taken in parts (a triangle's w lies in exactly
// one of them).  What bounds it is the walk: sum over the oriented edges
// u -> v of |out(v)| list words through L2, one or two shared-memory probes
// each; a warp waits for its lane with the longest chain of them, so tables are
// as sparse as the memory allows (an eighth or less filled up to 1,024 members;
// symmetric R-MAT 18: 710 us at a quarter, 544 so).
__global__ void __launch_bounds__(kThreads) k_tc_count(Store st, int n, const u32 *__restrict__ cnt,
                                                       const u32 *__restrict__ big, int per,
                                                       Ctl *c) {
  __shared__ __align__(16) u32 tab[kTabMax];
  __shared__ u32 s_u, s_pos;
  if (ld_cg_i32(&c->status) != 0) return;   // not symmetric (the same answer in every block)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u32 nlong = ld_cg_u32(&c->tc_nbig), nbig = nlong + ld_cg_u32(&c->tc_nmid);
  u64 sum = 0;
  // (what a block, and below a warp, takes first needs no counter: a small graph's
  // grid would queue up at one word to be told that nothing is left)
  for (bool first = true;; first = false) {
    __syncthreads();
    if (threadIdx.x == 0)
      s_u = first ? blockIdx.x : gridDim.x + atomicAdd(&c->tc_bpos, 1u);
    __syncthreads();
    if (s_u >= nbig) break;
    const u32 u = big[s_u < nlong ? s_u : (u32)n - 1u - (s_u - nlong)];
    const u32 d = cnt[u];
    const u32 *out = (const u32 *)(st.adj + st.alt[u]);
    // members per grab: every warp gets some, a lane each
    const u32 grab = min(32u, max(4u, (d + kThreads / 32 - 1) / (kThreads / 32)));
    for (u32 part = 0; part < d; part += kTabMax / 2) {
      const u32 np = min(d - part, kTabMax / 2);
      u32 bits = 7;
      while ((1u << bits) < 8 * np && (1u << bits) < kTabMax) ++bits;
      __syncthreads();
      for (u32 i = threadIdx.x; i < (1u << bits); i += kThreads) tab[i] = kEmpty;
      if (threadIdx.x == 0) s_pos = 0;
      __syncthreads();
      for (u32 i = threadIdx.x; i < np; i += kThreads) tab_put(tab, bits, out[part + i]);
      __syncthreads();
      for (;;) {
        u32 at = 0;
        if (lane == 0) at = atomicAdd(&s_pos, grab);
        at = __shfl_sync(kFull, at, 0);
        if (at >= d) break;
        const u32 i = at + lane;
        u32 len = 0;
        const u32 *p = nullptr;
        if (lane < (int)grab && i < d) {
          const u32 v = out[i];
          len = cnt[v];
          p = (const u32 *)(st.adj + st.alt[v]);
        }
        sum += count_lists(p, len, tab, bits);
      }
    }
  }
  __syncthreads();
  // short lists: a warp takes `per` vertices, then those with two members or more
  u32 *wtab = tab + warp * kWarpTab;
  const u32 gw = (u32)warp * gridDim.x + blockIdx.x, nw = gridDim.x * (kThreads / 32);
  for (bool first = true;; first = false) {
    u32 v0 = gw;
    if (!first && lane == 0) v0 = nw + atomicAdd(&c->tc_spos, 1u);
    const long long b = (long long)per * __shfl_sync(kFull, v0, 0);
    if (b >= n) break;
    const bool mine = lane < per && b + lane < n;
    const u32 dl = mine ? cnt[b + lane] : 0u;
    const long long al = mine ? st.alt[b + lane] : 0;
    u32 todo = __ballot_sync(kFull, dl >= 2 && dl <= kWarpList);
    while (todo) {
      const int o = __ffs(todo) - 1;
      todo &= todo - 1;
      const u32 d = __shfl_sync(kFull, dl, o);
      const u32 *out = (const u32 *)(st.adj + __shfl_sync(kFull, al, o));
#pragma unroll
      for (u32 k = 0; k < kWarpTab / 4; k += 32)
        ((uint4 *)wtab)[lane + k] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
      u32 len = 0;
      const u32 *p = nullptr;
      u32 v = 0;
      if ((u32)lane < d) {
        v = out[lane];
        len = cnt[v];
        p = (const u32 *)(st.adj + st.alt[v]);
      }
      __syncwarp();
      if ((u32)lane < d) tab_put(wtab, kWarpTabBits, v);
      __syncwarp();
      sum += count_lists(p, len, wtab, kWarpTabBits);
      __syncwarp();
    }
  }
  sum = warp_sum64(sum);
  if (lane == 0 && sum) atomicAdd(&c->tc_static, sum);
}

// First forward item in [lo, hi) whose key is at least `key`.
__device__ __forceinline__ long long item_lower(const u64 *keys, long long lo, long long hi,
                                                u64 key) {
  while (lo < hi) {
    const long long mid = (lo + hi) >> 1;
    if (__ldg(&keys[mid]) < key) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Is `key` an applied update among the sorted forward items [lo, hi)?
__device__ __forceinline__ bool item_applied(const u64 *keys, const unsigned char *flags,
                                             long long lo, long long hi, u64 key) {
  const long long end = hi;
  lo = item_lower(keys, lo, hi, key);
  // equal keys (repeated updates): the applied one may be any of them
  for (long long i = lo; i < end && __ldg(&keys[i]) == key; ++i)
    if (__ldg(&flags[i]) & 1) return true;
  return false;
}

// Every forward item has its reverse among the forward items (a thread per
// item); checked before anything changes.
__global__ void __launch_bounds__(kThreads) k_tc_batch_sym(const u64 *keys, long long nb, int bits,
                                                           Ctl *c) {
  const u64 cmask = (1ull << bits) - 1;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nb;
       i += (long long)gridDim.x * blockDim.x) {
    const u64 k = __ldg(&keys[i]);
    const u32 u = (u32)((k >> (bits + 1)) & cmask), v = (u32)((k >> 1) & cmask);
    const u64 r = ((u64)v << (bits + 1)) | ((u64)u << 1) | (k & 1);
    long long lo = 0, hi = nb;
    while (lo < hi) {
      const long long mid = (lo + hi) >> 1;
      if (__ldg(&keys[mid]) < r) lo = mid + 1; else hi = mid;
    }
    if (lo >= nb || __ldg(&keys[lo]) != r) atomicCAS(&c->status, 0, SP_EINVAL);
  }
}

// The corrections' work list.  Every updated pair is among the items in both
// directions and both see the same common neighbours with the same number of
// updated edges, so only u < v is walked and its sightings count twice
// (that both directions applied is counted here, for the host to check: a
// replayed batch can leave the graph with one direction of an edge).  An
// item whose shorter row is long is listed up to kMaxParts times, each part
// a share of the walk: without the split one pair of hubs (a walk of
// thousands of searches by one warp) outlasts the rest of the batch.
// Deletions are listed from the front of `tasks`, insertions from its end
// (2 nb words: at most nb / 2 pairs in all, kMaxParts of each).
constexpr int kMaxParts = 4;
constexpr int kPartWalk = 512;       // walked entries that make another part worth it

struct DeltaArgs {
  const u64 *keys;
  const unsigned char *flags;
  u64 *tasks;                        // item << 4 | parts - 1 << 2 | part
  long long nb, cap;
  int bits;
  Store st;
  Ctl *c;
};

__global__ void __launch_bounds__(kThreads) k_tc_tasks(DeltaArgs a) {
  if (ld_cg_i32(&a.c->status) != 0) return;
  const int lane = threadIdx.x & 31;
  const u64 cmask = (1ull << a.bits) - 1;
  const long long step = (long long)gridDim.x * kThreads;
  for (long long b = blockIdx.x * (long long)kThreads + (threadIdx.x & ~31); b < a.nb; b += step) {
    const long long i = b + lane;
    u32 parts[2] = {0, 0};
    int skew[2] = {0, 0};
    if (i < a.nb) {
      const u64 key = __ldg(&a.keys[i]);
      const u32 u = (u32)((key >> (a.bits + 1)) & cmask), v = (u32)((key >> 1) & cmask);
      const bool applied = __ldg(&a.flags[i]) & 1;
      if (applied && u != v) skew[key & 1] = u < v ? 1 : -1;
      if (u < v && applied) {
        const int du = __ldg(&a.st.row[u].deg), dv = __ldg(&a.st.row[v].deg);
        const int walk = du < dv ? du : dv;
        parts[key & 1] = (u32)min(kMaxParts, walk / kPartWalk + 1);
      }
    }
#pragma unroll
    for (int kind = 0; kind < 2; ++kind) {
      const int off = __reduce_add_sync(kFull, skew[kind]);
      if (lane == 0 && off) atomicAdd(&a.c->tc_skew[kind], off);
      const u32 incl = warp_incl_scan(parts[kind]), total = __shfl_sync(kFull, incl, 31);
      if (!total) continue;
      u64 base = 0;
      if (lane == 0) base = atomicAdd(&a.c->tc_ntask[kind], total);
      base = __shfl_sync(kFull, base, 0) + incl - parts[kind];
      for (u32 q = 0; q < parts[kind]; ++q) {
        const u64 at = base + q;
        if ((long long)at >= a.cap) {      // never expected: record and skip
          atomicExch(&a.c->bad, 1);
          break;
        }
        a.tasks[kind ? a.cap - 1 - at : at] = ((u64)i << 4) | ((u64)(parts[kind] - 1) << 2) | q;
      }
    }
  }
}

// The listing's correction for the listed updates of `kind` (a warp per task):
// sightings of common neighbours v3 by the number of updated edges of the
// triangle.  The warp walks its share of the shorter row, kDK entries per lane
// at a time, and searches the longer one with the lanes' searches in lockstep,
// so that kDK loads per lane are in flight at every level; a hit is looked up
// only among the batch items of rows v1 and v2, whose bounds are found once
// per task (four lanes at once), at its first hit (a sparse graph's tasks have
// hardly one: 60,000 pairs on 100,000 vertices, two batches, 534 -> 500 us).
// Bound by the searches' dependent levels through L2.  R-MAT 18, 1% of the pairs
// deleted and as many inserted: a batch 1.93 -> 0.54 ms against a warp per item
// over both directions, one search chain per lane, and every hit looked up among
// all items.
constexpr int kDK = 4;

__global__ void __launch_bounds__(kThreads) k_tc_delta(DeltaArgs a, int kind) {
  Ctl *c = a.c;
  if (ld_cg_i32(&c->status) != 0 || ld_cg_i32(&c->need_grow) != 0) return;
  const int lane = threadIdx.x & 31;
  const u64 cmask = (1ull << a.bits) - 1;
  const u64 ntask = ld_cg_u64(&c->tc_ntask[kind]);
  u64 k1 = 0, k2 = 0, k3 = 0;
  const u64 gw = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const u64 nw = gridDim.x * (kThreads / 32);
  for (bool first = true;; first = false) {   // (a warp's first task is that of its number)
    u64 t = gw;
    if (!first && lane == 0) t = nw + atomicAdd(&c->tc_tpos[kind], 1ull);
    t = __shfl_sync(kFull, t, 0);
    if (t >= ntask || (long long)t >= a.cap) break;
    const u64 task = __ldcg(&a.tasks[kind ? a.cap - 1 - t : t]);
    const u64 key = __ldg(&a.keys[task >> 4]);
    const int parts = (int)((task >> 2) & 3) + 1, part = (int)(task & 3);
    const u32 v1 = (u32)((key >> (a.bits + 1)) & cmask), v2 = (u32)((key >> 1) & cmask);
    const RowMeta r1 = a.st.row[v1], r2 = a.st.row[v2];
    const bool walk1 = r1.deg <= r2.deg;
    const int2 *wrow = a.st.adj + (walk1 ? r1.start : r2.start);
    const int wdeg = walk1 ? r1.deg : r2.deg;
    const int2 *srow = a.st.adj + (walk1 ? r2.start : r1.start);
    const int sdeg = walk1 ? r2.deg : r1.deg;
    long long bound = -1;
    for (int b = part * 32 * kDK; b < wdeg; b += parts * 32 * kDK) {
      int x[kDK], lo[kDK], hi[kDK];
#pragma unroll
      for (int k = 0; k < kDK; ++k) {
        const int e = b + 32 * k + lane;
        x[k] = e < wdeg ? __ldg(&wrow[e].x) : -1;
        lo[k] = 0;
        hi[k] = e < wdeg ? sdeg : 0;
      }
      // (halving: the rows of a batch's pairs are in L2, where the extra
      // arithmetic of an interpolating search costs more than its reads save)
      for (;;) {
        int y[kDK], mid[kDK];
        bool act = false;
#pragma unroll
        for (int k = 0; k < kDK; ++k) {
          act |= lo[k] < hi[k];
          mid[k] = (lo[k] + hi[k]) >> 1;
          y[k] = lo[k] < hi[k] ? __ldg(&srow[mid[k]].x) : 0;
        }
        if (!act) break;
#pragma unroll
        for (int k = 0; k < kDK; ++k)
          if (lo[k] < hi[k]) {
            if (y[k] < x[k]) lo[k] = mid[k] + 1; else hi[k] = mid[k];
          }
      }
      bool hit[kDK], any = false;
#pragma unroll
      for (int k = 0; k < kDK; ++k) {
        const u32 v3 = (u32)x[k];
        hit[k] = x[k] >= 0 && v3 != v1 && v3 != v2 && lo[k] < sdeg &&
                 __ldg(&srow[lo[k]].x) == x[k];
        any |= hit[k];
      }
      if (!__any_sync(kFull, any)) continue;
      if (__shfl_sync(kFull, bound, 0) < 0 && lane < 4) {
        // the batch items of rows v1 (lanes 0, 1) and v2 (lanes 2, 3)
        const u64 row = (u64)(lane < 2 ? v1 : v2) + (u64)(lane & 1);
        bound = item_lower(a.keys, 0, a.nb, row << (a.bits + 1));
      }
      __syncwarp();
      const long long lo1 = __shfl_sync(kFull, bound, 0), hi1 = __shfl_sync(kFull, bound, 1);
      const long long lo2 = __shfl_sync(kFull, bound, 2), hi2 = __shfl_sync(kFull, bound, 3);
#pragma unroll
      for (int k = 0; k < kDK; ++k) {
        if (!hit[k]) continue;
        const u32 v3 = (u32)x[k];
        const u64 tail = ((u64)v3 << 1) | (u64)kind;
        const int kk = 1 +
            item_applied(a.keys, a.flags, lo1, hi1, ((u64)v1 << (a.bits + 1)) | tail) +
            item_applied(a.keys, a.flags, lo2, hi2, ((u64)v2 << (a.bits + 1)) | tail);
        k1 += kk == 1;
        k2 += kk == 2;
        k3 += kk == 3;
      }
    }
  }
  k1 = warp_sum64(k1);
  k2 = warp_sum64(k2);
  k3 = warp_sum64(k3);
  if (lane == 0) {   // both directions of every pair
    u64 *dst = kind ? c->tc_ins : c->tc_del;
    if (k1) atomicAdd(&dst[0], 2 * k1);
    if (k2) atomicAdd(&dst[1], 2 * k2);
    if (k3) atomicAdd(&dst[2], 2 * k3);
  }
}

inline unsigned grid_for(long long work, int per_block, int cap) {
  long long b = (work + per_block - 1) / per_block;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (unsigned)b;
}

}  // namespace

// staticTC with the symmetry check: the count (or status SP_EINVAL) in ctl.
// Scratch: the forward store's alternate regions and the per-vertex words of
// the invalidation (g->jmp, g->cut, g->asv), all rewritten before their next
// use.
void launch_tc_static(sp_graph *g, int *launches) {
  OrientArgs a;
  a.fwd = g->fwd;
  a.rev = g->rev;
  a.cnt = g->jmp;
  a.giant = g->asv;
  a.c = g->ctl;
  a.n = g->n;
  const int warps = g->num_sms * 6 * (kThreads / 32);
  a.rpw = std::max(1, std::min(32, (int)(((long long)g->n + warps - 1) / warps)));
  k_tc_orient<<<grid_for(g->n, a.rpw * (kThreads / 32), g->num_sms * 16), kThreads, 0, g->stream>>>(
      a);
  ++*launches;
  // such a row takes two regions of that length (the host's edge count would not
  // do: it may lag behind the stores)
  if (g->fwd.slots > 2 * kOrientGiant) {
    k_tc_orient_giant<<<(unsigned)g->num_sms * 4, kThreads, 0, g->stream>>>(a);
    ++*launches;
  }
  k_tc_lists<<<grid_for(g->n, kThreads, g->num_sms * 8), kThreads, 0, g->stream>>>(a.cnt, g->n,
                                                                                   g->cut, g->ctl);
  // a small graph's vertices are spread over all warps: 32 of them one after the
  // other took 43 of the 74 us that 1,000 vertices' count was long
  const int per = std::max(1, std::min(32, (int)(g->n / (g->num_sms * 6 * (kThreads / 32)))));
  k_tc_count<<<(unsigned)g->num_sms * 6, kThreads, 0, g->stream>>>(g->fwd, g->n, a.cnt, g->cut,
                                                                   per, g->ctl);
  *launches += 2;
}

void launch_tc_batch_sym(sp_graph *g, long long nb, int *launches) {
  if (nb == 0) return;
  k_tc_batch_sym<<<grid_for(nb, kThreads, g->num_sms * 16), kThreads, 0, g->stream>>>(
      g->bb.keys, nb, g->bits, g->ctl);
  ++*launches;
}

static DeltaArgs delta_args(sp_graph *g, long long nb) {
  DeltaArgs a;
  a.keys = g->bb.keys;
  a.flags = g->bb.flags;
  a.tasks = g->bb.keys_alt;   // free once the sort has ended
  a.nb = nb;
  a.cap = 2 * nb;
  a.bits = g->bits;
  a.st = g->fwd;
  a.c = g->ctl;
  return a;
}

void launch_tc_tasks(sp_graph *g, long long nb, int *launches) {
  if (nb == 0) return;
  k_tc_tasks<<<grid_for(nb, kThreads, g->num_sms * 8), kThreads, 0, g->stream>>>(
      delta_args(g, nb));
  ++*launches;
}

void launch_tc_delta(sp_graph *g, long long nb, int kind, int *launches) {
  if (nb == 0) return;
  k_tc_delta<<<grid_for(nb * 32 * kMaxParts, kThreads, g->num_sms * 8), kThreads, 0, g->stream>>>(
      delta_args(g, nb), kind);
  ++*launches;
}

}  // namespace sp
