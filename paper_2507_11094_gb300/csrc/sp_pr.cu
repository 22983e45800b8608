// sp_pr.cu -- dynamic PageRank (paper, appendix listing "Dynamic PR coded in
// StarPlat DSL": staticPR, Decremental, Incremental): the Jacobi steps over
// the vertices of a phase (all of them, or those that propagateNodeFlags
// flagged), in one cooperative launch.
//
// A step needs, for every selected v, the sum of pr[u] / outdeg(u) over the
// in-edges u -> v.  Its floor is one read of the in-edge list; what it pays
// for instead is the gather, one 4-byte term from a random place per edge:
// a warp's 32 terms lie on 32 cache lines, which the L1 serves one per clock
// (55 us for 16.8 M edges), and every miss moves a 32-byte sector out of L2.
// So the launch first prepares what all its steps share:
//   * the terms of the kHot vertices with the most out-edges get the first
//     places of the term array, and every step starts by copying those into
//     shared memory, where a gather costs a bank conflict or two instead of
//     a line each (on R-MAT 20 they serve about three quarters of the edges);
//   * each selected vertex's in-neighbours are written as plain u32 places,
//     one list after the other, padded to whole 16-byte loads with a place
//     that holds zero: half the bytes of the (col, w) pairs without the
//     store's slack, so that most of them stay in L2 from step to step (left
//     in the rows' alternate regions, which is where they go when there is no
//     room for them, R-MAT 20's 67 MB cost 149 MB of HBM reads a step);
//   * the vertices are listed by in-degree class, with everything a step
//     needs of one in arrays over its position in that list; a term's place,
//     where it is not hot, follows its vertex's position.
// A step then reads its lists once: the warps of a block take units of work as
// they come (a segment, a row, four rows, 32 rows, two units read ahead) from
// the block's equal share of the words, the sums meet in shared memory, and
// the rows are finished 32 consecutive positions to a warp.  Finishing each
// row by the lane that had its sum cost 117 of 168 us a step on R-MAT 20 (half
// a million scattered 4-byte stores, which the L2's halves pass back and
// forth, and 64-bit adds for one lane each); a fixed share of the rows per
// warp left 25-40 us of a step waiting.  No accumulator array, no atomics on
// ranks, one grid barrier a step.  Only a row of more than kSegLen in-edges is
// cut into segments; the warp that ends its last one adds the parts up, in
// order, so a step's sums do not depend on the schedule.
//
// sp_pr_init on R-MAT 20 (16.8 M edges, 50 steps): 7.35 -> 3.34 ms, a step
// 143 -> 62 us (edge chunks over (col, w) pairs, per-edge L2 gathers, float
// atomics into an accumulator and two barriers before).  Now bound by the
// cold gathers and the list reads through L2, about half each.
#include <algorithm>

#include "sp_acc.cuh"
#include "sp_loop.cuh"

namespace sp {

namespace {

constexpr int kPrThreads = 1024;
constexpr u32 kHot = 28160;              // places in shared memory: 110 KB
constexpr u32 kZeroPlace = kHot;         // always 0: the padding of the lists
constexpr u32 kPrBins = 1024;            // out-degree bins (the last: and above)
static_assert(kPrBins == kPrThreads, "one bin per thread");
constexpr u32 kRowTile = 4096;           // rows a block sums before it finishes them
// (with the static part just below 132 KB: the next larger split of an SM's
// memory leaves the L1 too few lines for a full block's gathers)
constexpr size_t kPrSmem = (size_t)(kHot + 4 + kRowTile) * sizeof(float);
// in-degree classes: a row of more than kSegLen in-edges in segments of that
// length, a warp each; down to kGroupMax a warp; down to kLaneMax eight
// lanes; the rest a lane; rows without in-edges take the constant term in every
// step.  The vertices of no phase come last.
constexpr u32 kSegLen = 1024, kGroupMax = 64, kLaneMax = 8;
enum { kClsHub = 0, kClsWarp, kClsGroup, kClsLane, kClsZero, kClsOut, kClasses };

// Zeroed before every launch.
struct PrScratch {
  u32 bins[kPrBins];     // vertices by out-degree
  u64 cls[kClasses];     // per class: vertices << 32 | 16-byte words of their lists
  u64 edges;             // in-edges of the selected vertices
  u32 segs;              // segments of the longest rows
  u32 hot;               // hot places handed out
};

struct PrArgs {
  Ctl *ctl;
  Limits lim;
  Store fwd, rev;
  PrScratch *sc;
  u32 *lists;            // room for the packed in-neighbour lists, or null
  u64 list_words;        // ... in 16-byte words
  float *pr;             // ranks by vertex
  float *term[2];        // pr / outdeg by place (kHot, the zero place, then by vertex)
  u32 *place;            // a vertex's place
  const u32 *flag;       // selected: all, or flag[v] == tag
  u32 tag;
  int all;
  float init;            // all: every rank starts at this
  // by position in the class order
  u64 *list;             // where the in-neighbour list starts in `lists`
  int2 *lenp;            // list length, place
  int2 *degv;            // out-degree, vertex
  float *rank;
  u32 *segbase, *segleft;   // rows in segments: first segment, segments done
  u32 *seg;              // by segment: its row's position
  float *part;           // ... and its sum
  int n;
  float base, damping;
  double beta;
  int max_iter;
};

__device__ __forceinline__ double *prd_ptr(Ctl *c, u32 b) {
  return b == 0 ? &c->prd0 : (b == 1 ? &c->prd1 : &c->prd2);
}

__device__ __forceinline__ int in_class(u32 d) {
  return d > kSegLen ? kClsHub : d > kGroupMax ? kClsWarp : d > kLaneMax ? kClsGroup
         : d > 0 ? kClsLane : kClsZero;
}

__device__ __forceinline__ float term_of(float rank, int outdeg) {
  return outdeg > 0 ? __fdiv_rn(rank, (float)outdeg) : 0.0f;
}

// The term at place p: from shared memory where it is hot, else from L2.  Both
// loads are issued without a branch (a lane whose term is not hot reads the
// zero place, one whose term is hot skips the global load), so that all the
// gathers of a lane are in flight together; with a branch per place each one
// waited for the one before it.
__device__ __forceinline__ float cold_term(const float *term, u32 p) {
  float r;
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.gt.u32 q, %2, %3;\n\tmov.f32 %0, 0f00000000;\n\t"
      "@q ld.global.cg.f32 %0, [%1];\n\t}"
      : "=f"(r)
      : "l"(term + p), "r"(p), "n"(kZeroPlace));
  return r;
}

__device__ __forceinline__ u32 atom_add_acq_rel(u32 *p, u32 x) {
  u32 r;
  asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(r) : "l"(p), "r"(x) : "memory");
  return r;
}

// The terms of U words of four places each (x + 0 is exact).
template <int U>
__device__ __forceinline__ void gather(const float *hot, const float *term, const uint4 *w,
                                       float4 *f) {
  float4 g[U];
#pragma unroll
  for (int k = 0; k < U; ++k) {
    g[k].x = cold_term(term, w[k].x);
    g[k].y = cold_term(term, w[k].y);
    g[k].z = cold_term(term, w[k].z);
    g[k].w = cold_term(term, w[k].w);
  }
#pragma unroll
  for (int k = 0; k < U; ++k) {
    f[k].x = hot[min(w[k].x, kZeroPlace)] + g[k].x;
    f[k].y = hot[min(w[k].y, kZeroPlace)] + g[k].y;
    f[k].z = hot[min(w[k].z, kZeroPlace)] + g[k].z;
    f[k].w = hot[min(w[k].w, kZeroPlace)] + g[k].w;
  }
}

// Sum of the lane's share of a list: 16-byte words q0, q0 + stride, ... below
// nq, U of them in flight.
template <int U>
__device__ __forceinline__ float sum_words(const float *hot, const float *term, const uint4 *l,
                                           u32 q0, u32 nq, u32 stride) {
  const uint4 pad = make_uint4(kZeroPlace, kZeroPlace, kZeroPlace, kZeroPlace);
  float s = 0.0f;
  for (u32 q = q0; q < nq; q += U * stride) {
    uint4 w[U];
    float4 f[U];
#pragma unroll
    for (int k = 0; k < U; ++k) w[k] = q + k * stride < nq ? __ldcg(l + q + k * stride) : pad;
    gather<U>(hot, term, w, f);
#pragma unroll
    for (int k = 0; k < U; ++k) s += (f[k].x + f[k].y) + (f[k].z + f[k].w);
  }
  return s;
}

// A unit of a step's work for one warp: every lane's list, the word it starts
// at, the lanes that share the list, and the row the sum belongs to.
struct Unit {
  const uint4 *l;
  u32 nq, q0, width, row, u;
};

// What a tile's units are: segments, then rows of a warp, of eight lanes, of a
// lane (ends of the unit numbers, and the rows of each).
struct Tile {
  u32 segs, uw, ug, ul, w0, w1, g0, g1, l0, l1;
};

__device__ __forceinline__ void first_words(const Unit &x, uint4 w[2]) {
  const uint4 pad = make_uint4(kZeroPlace, kZeroPlace, kZeroPlace, kZeroPlace);
  w[0] = x.q0 < x.nq ? __ldcg(x.l + x.q0) : pad;
  w[1] = x.q0 + x.width < x.nq ? __ldcg(x.l + x.q0 + x.width) : pad;
}

// The new rank of the row at a position from the sum of its terms.
__device__ __forceinline__ void finish(const PrArgs &a, float *next, u32 pos, float sum, int place,
                                       int outdeg, float old, Acc &diff) {
  const float val = __fadd_rn(a.base, __fmul_rn(a.damping, sum));
  acc_diff(diff, val, old);
  __stcg(a.rank + pos, val);
  __stcg(next + place, term_of(val, outdeg));
}

// Write the lane's share of one vertex's list (words of four places).
__device__ __forceinline__ void write_list(const PrArgs &a, long long start, u32 len, u32 *list,
                                           u32 q0, u32 nq, u32 stride) {
  uint4 *l = (uint4 *)list;
  for (u32 q = q0; q < nq; q += stride) {
    int x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = 4 * q + k < len ? __ldg(&a.rev.adj[start + 4 * q + k].x) : -1;
    u32 p[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) p[k] = x[k] >= 0 ? __ldcg(a.place + x[k]) : kZeroPlace;
    __stcg(l + q, make_uint4(p[0], p[1], p[2], p[3]));
  }
}

__global__ void __launch_bounds__(kPrThreads, 1) k_pr(PrArgs a) {
  extern __shared__ __align__(16) float hot[];
  __shared__ u32 scratch[40];
  __shared__ u64 s_cls[kClasses];
  __shared__ u32 s_segs, s_T, s_hot, s_nhot, s_unit, s_lo[3], s_hi[3];
  __shared__ double s_sum[kPrThreads / 32];
  Ctl *c = a.ctl;
  if (!repair_enabled_block(c)) return;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const u32 n = (u32)a.n, G = gridDim.x;
  constexpr int kF = kRowTile / kPrThreads;   // rows that a thread takes at a time
  const u32 chunk = (n + G - 1) / G;
  const u32 cb = min(blockIdx.x * chunk, n), ce = min(cb + chunk, n);
  u64 *bar = &c->bar_push;
  u64 target = 0;
  float *s_row = hot + kHot + 4;
  u32 *s_bins = (u32 *)hot;      // the preparation uses the hot places' memory

  // 1. out-degree bins of all vertices, class counts of the selected ones
  s_bins[t] = 0;
  if (t < kClasses) s_cls[t] = 0;
  if (t == 0) s_segs = 0;
  __syncthreads();
  u64 edges = 0;
  for (u32 b = cb + (t & ~31); b < ce; b += kF * kPrThreads) {
    u32 od[kF], id[kF], fl[kF];
#pragma unroll
    for (int q = 0; q < kF; ++q) {   // kF vertices' loads in flight together
      const u32 v = b + q * kPrThreads + lane;
      const bool on = v < ce;
      fl[q] = on && !a.all ? __ldcg(a.flag + v) : a.tag;
      od[q] = on ? (u32)__ldg(&a.fwd.row[v].deg) : 0u;
      id[q] = on ? (u32)__ldg(&a.rev.row[v].deg) : 0u;
    }
#pragma unroll
    for (int q = 0; q < kF; ++q) {
      const bool on = b + q * kPrThreads + lane < ce, sel = on && fl[q] == a.tag;
      if (!sel) id[q] = 0;
      if (on) atomicAdd(&s_bins[min(od[q], kPrBins - 1)], 1u);
      const int cls = sel ? in_class(id[q]) : on ? kClsOut : -1;
#pragma unroll
      for (int k = 0; k < kClasses; ++k) {
        const u32 m = __ballot_sync(kFull, cls == k);
        if (!m) continue;
        const u32 w = __reduce_add_sync(kFull, cls == k ? (id[q] + 3) / 4 : 0u);
        if (lane == 0) atomicAdd(&s_cls[k], ((u64)__popc(m) << 32) | w);
      }
      if (cls == kClsHub) atomicAdd(&s_segs, (id[q] + kSegLen - 1) / kSegLen);
      edges += id[q];
    }
  }
  edges = warp_sum(edges);
  if (lane == 0 && edges) atomicAdd(&a.sc->edges, edges);
  __syncthreads();
  const u32 mybin = s_bins[t];
  if (mybin) atomicAdd(&a.sc->bins[t], mybin);
  // the block's ranges inside each class (their order does not matter;
  // positions and words are handed out together, so lists lie in the order of
  // the positions)
  if (t < kClasses) s_cls[t] = s_cls[t] ? atomicAdd(&a.sc->cls[t], s_cls[t]) : 0ull;
  if (t == 32) s_segs = s_segs ? atomicAdd(&a.sc->segs, s_segs) : 0u;
  target += G;
  bool stop = grid_sync(bar, target, c, a.lim);

  // 2. the out-degree from which a vertex is hot, every vertex's place and
  // term, and the selected vertices by position
  u32 first[kClasses], cnt[kClasses];
  const u32 nsegs = __ldcg(&a.sc->segs);
  bool packed;
  {
    u64 at = 0;
#pragma unroll
    for (int k = 0; k < kClasses; ++k) {
      const u64 x = ld_cg_u64(&a.sc->cls[k]);
      cnt[k] = (u32)(x >> 32);
      first[k] = (u32)(at >> 32);
      if (t == k) s_cls[k] += at;
      at += x;
    }
    // packed, if the rows as they are now fit: the room follows the host's edge
    // count, which an asynchronous batch that nobody finished leaves behind (the
    // same answer in every block: the counts are final since the barrier)
    packed = a.lists && (u64)(u32)at <= a.list_words;
    if (t == 0) {
      s_T = kPrBins;
      s_hot = 0;
    }
    // thread t looks at bin kPrBins - 1 - t: the vertices above it
    const u32 d = kPrBins - 1 - (u32)t;
    u32 total;
    const u32 here = d > 0 ? __ldcg(&a.sc->bins[d]) : 0u;
    const u32 above = block_excl_scan(here, scratch, &total);
    if (d > 0 && above < kHot) atomicMin(&s_T, d);
    if (t == 0) s_nhot = min(total, kHot);
    __syncthreads();
    // the block's hot places
    const u32 mine = (u32)t >= s_T ? mybin : 0u;
    block_excl_scan(mine, scratch, &total);
    if (t == 0) s_hot = total ? atomicAdd(&a.sc->hot, total) : 0u;
    __syncthreads();
  }
  u32 *lists = packed ? a.lists : (u32 *)a.rev.adj;
  const u32 T = s_T, nhot = s_nhot;
  u32 nfl = a.tag;   // the next vertex's flag, out-degree and rank, read one ahead
  int nod = 0;
  float nr = a.init;
  auto ahead = [&](u32 v) {
    if (v >= ce) return;
    nod = __ldg(&a.fwd.row[v].deg);
    if (!a.all) {
      nfl = __ldcg(a.flag + v);
      nr = __ldcg(a.pr + v);
    }
  };
  ahead(cb + t);
  for (u32 b = cb + (t & ~31); b < ce && !stop; b += kPrThreads) {
    const u32 v = b + lane;
    const bool on = v < ce;
    const bool sel = on && nfl == a.tag;
    const int od = on ? nod : 0;
    const float r = on ? nr : 0.0f;
    const RowMeta in = sel ? a.rev.row[v] : RowMeta{0, 0, 0};
    ahead(v + kPrThreads);
    const int cls = sel ? in_class((u32)in.deg) : on ? kClsOut : -1;
    u32 pos = 0, wpos = 0;
    const u32 nw4 = ((u32)in.deg + 3) / 4;
#pragma unroll
    for (int k = 0; k < kClasses; ++k) {
      const u32 m = __ballot_sync(kFull, cls == k);
      if (!m) continue;
      const u32 wi = warp_incl_scan(cls == k ? nw4 : 0u);
      u64 base = 0;
      if (lane == 31) base = atomicAdd(&s_cls[k], ((u64)__popc(m) << 32) | wi);
      base = __shfl_sync(kFull, base, 31);
      if (cls == k) {
        pos = (u32)(base >> 32) + __popc(m & lanemask_lt());
        wpos = (u32)base + wi - nw4;
      }
    }
    u32 p = kHot + 1 + pos;
    {
      const bool h = on && (u32)od >= T;
      const u32 m = __ballot_sync(kFull, h);
      u32 base = 0;
      if (lane == 0 && m) base = atomicAdd(&s_hot, (u32)__popc(m));
      base = __shfl_sync(kFull, base, 0) + __popc(m & lanemask_lt());
      if (h && base < kHot) p = base;
    }
    if (on) {
      const float f = term_of(r, od);
      a.place[v] = p;
      a.term[0][p] = f;
      a.term[1][p] = f;
    }
    if (sel) {
      a.list[pos] = packed ? 4ull * wpos : 2ull * (u64)a.rev.alt[v];
      a.lenp[pos] = make_int2(in.deg, (int)p);
      a.degv[pos] = make_int2(od, (int)v);
      a.rank[pos] = r;
      if (cls == kClsHub) {
        const u32 ns = ((u32)in.deg + kSegLen - 1) / kSegLen;
        const u32 sb = atomicAdd(&s_segs, ns);
        a.segbase[pos] = sb;
        a.segleft[pos] = 0;
        for (u32 k = 0; k < ns; ++k) a.seg[sb + k] = pos;
      }
    }
  }
  if (t < 4) hot[kZeroPlace + t] = 0.0f;
  if (t == 0) s_unit = 0;
  target += G;
  if (!stop) stop = grid_sync(bar, target, c, a.lim);

  // the block's rows: per class the positions whose lists start in its share
  // of the class's words (lists in the alternate regions: its share of the
  // positions)
  if (!stop && t < 6) {
    const int k = kClsWarp + t % 3;
    const u32 b = blockIdx.x + t / 3;
    u32 r = (u32)((u64)cnt[k] * b / G);
    if (packed && b > 0 && b < G && cnt[k] > 0) {
      const u64 w0 = __ldcg(a.list + first[k]);
      const u64 want = w0 + 4 * ((u64)(u32)ld_cg_u64(&a.sc->cls[k]) * b / G);
      u32 lo = 0, hi = cnt[k];
      while (lo < hi) {
        const u32 mid = (lo + hi) >> 1;
        if (__ldcg(a.list + first[k] + mid) < want) lo = mid + 1; else hi = mid;
      }
      r = lo;
    }
    (t < 3 ? s_lo : s_hi)[t % 3] = r;
  }
  __syncthreads();
  u32 row0[3], rows[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    row0[k] = first[kClsWarp + k] + s_lo[k];
    rows[k] = stop ? 0u : s_hi[k] - s_lo[k];
  }
  const u32 nrow = rows[0] + rows[1] + rows[2];

  // 3. the in-neighbour lists, each by the block that will read it
  const u32 mysegs = nsegs > blockIdx.x ? (nsegs - blockIdx.x + G - 1) / G : 0u;
  if (!stop) {
    for (u32 j = warp; j < mysegs; j += kPrThreads / 32) {
      const u32 i = blockIdx.x + j * G, pos = __ldcg(a.seg + i);
      const u32 len = (u32)__ldcg(&a.lenp[pos].x), at = (i - __ldcg(a.segbase + pos)) * kSegLen;
      const u32 v = (u32)__ldcg(&a.degv[pos].y);
      const u32 sl = min(kSegLen, len - at);
      write_list(a, a.rev.row[v].start + at, sl, lists + __ldcg(a.list + pos) + at, lane,
                 (sl + 3) / 4, 32);
    }
    for (u32 i = warp; i < rows[0]; i += kPrThreads / 32) {
      const u32 pos = row0[0] + i;
      const u32 len = (u32)__ldcg(&a.lenp[pos].x), v = (u32)__ldcg(&a.degv[pos].y);
      write_list(a, a.rev.row[v].start, len, lists + __ldcg(a.list + pos), lane, (len + 3) / 4, 32);
    }
    for (u32 i = t >> 3; i < rows[1]; i += kPrThreads / 8) {
      const u32 pos = row0[1] + i;
      const u32 len = (u32)__ldcg(&a.lenp[pos].x), v = (u32)__ldcg(&a.degv[pos].y);
      write_list(a, a.rev.row[v].start, len, lists + __ldcg(a.list + pos), lane & 7, (len + 3) / 4, 8);
    }
    for (u32 i = t; i < rows[2]; i += kPrThreads) {
      const u32 pos = row0[2] + i;
      const u32 len = (u32)__ldcg(&a.lenp[pos].x), v = (u32)__ldcg(&a.degv[pos].y);
      write_list(a, a.rev.row[v].start, len, lists + __ldcg(a.list + pos), 0, (len + 3) / 4, 1);
    }
  }
  __syncthreads();

  // a block's share of k positions: one run of them
  auto share = [&](u32 k, u32 b) { return (u32)((u64)k * b / G); };
  // 4. Jacobi steps
  u32 it = 0, cur = 0;
  for (;;) {
    if (stop) break;
    const float *term = a.term[cur];
    float *next = a.term[cur ^ 1];
    for (u32 i = t; i < (nhot + 3) / 4; i += kPrThreads)
      ((float4 *)hot)[i] = __ldcg((const float4 *)term + i);
    __syncthreads();
    if (blockIdx.x == 0 && t == 0) *(volatile double *)prd_ptr(c, (it + 1) % 3) = 0.0;
    Acc diff;
    // sums into shared memory by whichever lanes suit the row, in units that
    // the warps take as they come: a segment, a row, four rows, 32 rows
    for (u32 r0 = 0; r0 == 0 || r0 < nrow; r0 += kRowTile) {
      const u32 r1 = min(r0 + kRowTile, nrow);
      Tile tl;
      tl.segs = r0 == 0 ? mysegs : 0u;
      tl.w0 = min(r0, rows[0]);
      tl.w1 = min(r1, rows[0]);
      tl.g0 = min(max(r0, rows[0]), rows[0] + rows[1]);
      tl.g1 = min(max(r1, rows[0]), rows[0] + rows[1]);
      tl.l0 = max(r0, rows[0] + rows[1]);
      tl.l1 = max(r1, rows[0] + rows[1]);
      tl.uw = tl.segs + (tl.w1 - tl.w0);
      tl.ug = tl.uw + (tl.g1 - tl.g0 + 3) / 4;
      tl.ul = tl.ug + (tl.l1 - tl.l0 + 31) / 32;
      auto grab = [&]() {
        u32 u = 0;
        if (lane == 0) u = atomicAdd(&s_unit, 1u);
        return __shfl_sync(kFull, u, 0);
      };
      auto load = [&](u32 u) {
        Unit x;
        x.u = u;
        x.q0 = (u32)lane;
        x.width = 32;
        x.row = ~0u;
        x.l = nullptr;
        x.nq = 0;
        if (u < tl.segs) {
          const u32 i = blockIdx.x + u * G, pos = __ldcg(a.seg + i);
          const u32 at = (i - __ldcg(a.segbase + pos)) * kSegLen;
          x.l = (const uint4 *)(lists + __ldcg(a.list + pos) + at);
          x.nq = (min(kSegLen, (u32)__ldcg(&a.lenp[pos].x) - at) + 3) / 4;
          return x;
        }
        u32 pos = 0;
        if (u < tl.uw) {
          x.row = tl.w0 + (u - tl.segs);
          pos = row0[0] + x.row;
        } else if (u < tl.ug) {
          x.width = 8;
          x.q0 = lane & 7;
          const u32 i = tl.g0 + 4 * (u - tl.uw) + (lane >> 3);
          if (i < tl.g1) {
            x.row = i;
            pos = row0[1] + (i - rows[0]);
          }
        } else if (u < tl.ul) {
          x.width = 1;
          x.q0 = 0;
          const u32 i = tl.l0 + 32 * (u - tl.ug) + lane;
          if (i < tl.l1) {
            x.row = i;
            pos = row0[2] + (i - rows[0] - rows[1]);
          }
        }
        if (x.row != ~0u) {
          x.l = (const uint4 *)(lists + __ldcg(a.list + pos));
          x.nq = ((u32)__ldcg(&a.lenp[pos].x) + 3) / 4;
        }
        return x;
      };
      // two units ahead: a unit's list address and its first words are two
      // dependent reads that would otherwise stand in front of its gathers
      Unit x0 = load(grab()), x1 = load(grab());
      uint4 w0[2], w1[2];
      first_words(x0, w0);
      while (x0.u < tl.ul) {
        const Unit x2 = load(grab());
        first_words(x1, w1);
        float4 f[2];
        gather<2>(hot, term, w0, f);
        float x = ((f[0].x + f[0].y) + (f[0].z + f[0].w)) + ((f[1].x + f[1].y) + (f[1].z + f[1].w));
        if (2 * x0.width < x0.nq)
          x += sum_words<2>(hot, term, x0.l, x0.q0 + 2 * x0.width, x0.nq, x0.width);
        for (u32 o = x0.width / 2; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
        if (x0.row != ~0u && x0.q0 == 0) s_row[x0.row - r0] = x;
        if (x0.u < tl.segs) {
          const u32 i = blockIdx.x + x0.u * G, pos = __ldcg(a.seg + i);
          const int2 lp = __ldcg(a.lenp + pos);
          const u32 sb = __ldcg(a.segbase + pos), nseg = ((u32)lp.x + kSegLen - 1) / kSegLen;
          u32 last = 0;
          if (lane == 0) {
            __stcg(a.part + i, x);
            last = atom_add_acq_rel(a.segleft + pos, 1u) == nseg - 1;
          }
          last = __shfl_sync(kFull, last, 0);
          __syncwarp();
          if (last) {   // the row's last segment: its parts, in order
            float y = 0.0f;
            for (u32 k = lane; k < nseg; k += 32) y += __ldcg(a.part + sb + k);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) y += __shfl_xor_sync(kFull, y, o);
            if (lane == 0) {
              __stcg(a.segleft + pos, 0u);
              finish(a, next, pos, y, lp.y, __ldcg(&a.degv[pos].x), __ldcg(a.rank + pos), diff);
            }
          }
        }
        x0 = x1;
        x1 = x2;
        w0[0] = w1[0];
        w0[1] = w1[1];
      }
      __syncthreads();
      if (t == 0) s_unit = 0;
      // then a thread per row finishes them, so that ranks and terms go 32
      // consecutive positions to a warp
      u32 pos[kF];
      int p[kF], od[kF];
      float rk[kF];
#pragma unroll
      for (int k = 0; k < kF; ++k) {
        const u32 i = r0 + k * kPrThreads + t;
        pos[k] = i < rows[0]             ? row0[0] + i
                 : i < rows[0] + rows[1] ? row0[1] + (i - rows[0])
                                         : row0[2] + (i - rows[0] - rows[1]);
        if (i < r1) {
          p[k] = __ldcg(&a.lenp[pos[k]].y);
          od[k] = __ldcg(&a.degv[pos[k]].x);
          rk[k] = __ldcg(a.rank + pos[k]);
        }
      }
#pragma unroll
      for (int k = 0; k < kF; ++k)
        if (r0 + k * kPrThreads + t < r1)
          finish(a, next, pos[k], s_row[k * kPrThreads + t], p[k], od[k], rk[k], diff);
      __syncthreads();
    }
    // no in-edges: the constant term, from the first step on (and into both
    // term buffers); kF rows' loads together (10 M such rows: 450 us a step when
    // each waited alone, 85 so)
    if (it < 2) {
      const u32 z1 = first[kClsZero] + share(cnt[kClsZero], blockIdx.x + 1);
      for (u32 z0 = first[kClsZero] + share(cnt[kClsZero], blockIdx.x); z0 < z1;
           z0 += kF * kPrThreads) {
        int p[kF], od[kF];
        float rk[kF];
#pragma unroll
        for (int k = 0; k < kF; ++k) {
          const u32 pos = z0 + k * kPrThreads + t;
          if (pos < z1) {
            p[k] = __ldcg(&a.lenp[pos].y);
            od[k] = __ldcg(&a.degv[pos].x);
            rk[k] = __ldcg(a.rank + pos);
          }
        }
#pragma unroll
        for (int k = 0; k < kF; ++k)
          if (z0 + k * kPrThreads + t < z1)
            finish(a, next, z0 + k * kPrThreads + t, 0.0f, p[k], od[k], rk[k], diff);
      }
    }
    {
      // (the warp's 32 sums meet as floats too: in 64 bits 1.8 us a step)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        Acc other;
        other.hi = __shfl_xor_sync(kFull, diff.hi, o);
        other.mid = __shfl_xor_sync(kFull, diff.mid, o);
        other.lo = __shfl_xor_sync(kFull, diff.lo, o);
        acc_merge(diff, other);
      }
      if (lane == 0) s_sum[warp] = acc_value(diff);
      __syncthreads();
      if (warp == 0) {
        double x = s_sum[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
        if (lane == 0 && x != 0.0) atomicAdd(prd_ptr(c, it % 3), x);
      }
    }
    target += G;
    stop = grid_sync(bar, target, c, a.lim);
    if (stop) break;
    const double d = *(volatile double *)prd_ptr(c, it % 3);
    ++it;
    cur ^= 1;
    if (!(d > a.beta) || it >= (u32)a.max_iter) break;
  }
  if (!stop) {
    const u32 all = first[kClsZero] + cnt[kClsZero], i1 = share(all, blockIdx.x + 1);
    for (u32 i = share(all, blockIdx.x) + t; i < i1; i += kPrThreads)
      a.pr[(u32)__ldcg(&a.degv[i].y)] = __ldcg(a.rank + i);
  }
  if (blockIdx.x == 0 && t == 0) {
    volatile Ctl *vc = c;
    vc->pull_edges = (u64)it * __ldcg(&a.sc->edges);
    vc->pr_iters = it;
    vc->rounds_push = it;
  }
}

}  // namespace

// The PageRank buffers of a handle (all of them, or none on SP_ENOMEM).
sp_status pr_alloc(sp_graph *g) {
  if (g->pr) return SP_OK;
  if (cudaFuncSetAttribute(k_pr, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPrSmem) !=
      cudaSuccess)
    return SP_ECUDA;
  const size_t nn = (size_t)g->n;
  const size_t sz[6] = {nn * 4, (nn + kHot + 1) * 4, (nn + kHot + 1) * 4, nn * 4, nn * 4,
                        sizeof(PrScratch)};
  void *p[6];
  bool ok = true;
  for (int i = 0; i < 6; ++i) {
    p[i] = ok ? g->al.get(sz[i]) : nullptr;
    ok = ok && p[i];
  }
  if (!ok) {
    for (int i = 0; i < 6; ++i) g->al.put(p[i], sz[i]);
    return SP_ENOMEM;
  }
  g->pr = (float *)p[0];
  g->prterm[0] = (float *)p[1];
  g->prterm[1] = (float *)p[2];
  g->prplace = (u32 *)p[3];
  g->prflag = (u32 *)p[4];
  g->prscratch = p[5];
  cudaMemsetAsync(g->prflag, 0, nn * 4, g->stream);
  g->prtag = 0;
  return SP_OK;
}

void pr_free(sp_graph *g) {
  const size_t nn = (size_t)g->n;
  g->al.put(g->pr, nn * 4);
  g->al.put(g->prterm[0], (nn + kHot + 1) * 4);
  g->al.put(g->prterm[1], (nn + kHot + 1) * 4);
  g->al.put(g->prplace, nn * 4);
  g->al.put(g->prflag, nn * 4);
  g->al.put(g->prscratch, sizeof(PrScratch));
  if (g->prlist) g->al.put(g->prlist, g->prlist_bytes);
}

// Room for the packed lists of m edges (a row's list is padded by up to three
// places); without it the lists go to the alternate regions.
static void pr_lists(sp_graph *g) {
  const long long rows = std::min<long long>(g->n, g->m);
  const size_t need = 4 * (size_t)(g->m + 3 * rows) + 16;
  if (need <= g->prlist_bytes) return;
  const size_t bytes = need + need / 8;
  void *p = g->al.get(bytes);
  if (g->prlist) g->al.put(g->prlist, g->prlist_bytes);
  g->prlist = (u32 *)p;
  g->prlist_bytes = p ? bytes : 0;
}

// The Jacobi steps of a phase: over all vertices, each starting at `init`, or
// over the flagged ones.  Scratch (rewritten by its owners before their next
// use): the frontier queues' arrays, the invalidation's words, the
// chunk-owner tables and the reverse store's alternate regions.
cudaError_t launch_pr(sp_graph *g, int all, float init, int *launches) {
  pr_lists(g);
  PrArgs p;
  p.lists = g->prlist;
  p.list_words = g->prlist_bytes / 16;
  p.ctl = g->ctl;
  p.lim = g->lim;
  p.fwd = g->fwd;
  p.rev = g->rev;
  p.sc = (PrScratch *)g->prscratch;
  p.pr = g->pr;
  p.term[0] = g->prterm[0];
  p.term[1] = g->prterm[1];
  p.place = g->prplace;
  p.flag = g->prflag;
  p.tag = g->prtag;
  p.all = all;
  p.init = init;
  p.list = (u64 *)g->qent[0];
  p.lenp = g->qent[1];
  p.degv = g->qent[2];
  p.rank = (float *)g->jmp;
  p.segbase = g->cut;
  p.segleft = g->asv;
  // a row of d > kSegLen in-edges has at most 2 d / kSegLen segments, and the
  // chunk-owner tables hold a word per kChunk of its 2 d slots
  static_assert(kSegLen >= (u32)kChunk, "the segments fit the chunk-owner tables");
  p.seg = g->qown[0];
  p.part = (float *)g->qown[1];
  p.n = g->n;
  p.base = (1.0f - g->pr_damping) / (float)g->n;
  p.damping = g->pr_damping;
  p.beta = (double)g->pr_beta;
  p.max_iter = g->pr_max_iter;
  cudaMemsetAsync(g->prscratch, 0, sizeof(PrScratch), g->stream);
  int blocks = g->num_sms;
  if (g->loop_blocks_user > 0 && g->loop_blocks_user < blocks) blocks = g->loop_blocks_user;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(kPrThreads);
  cfg.dynamicSmemBytes = kPrSmem;
  cfg.stream = g->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  ++*launches;
  return cudaLaunchKernelEx(&cfg, k_pr, p);
}

}  // namespace sp
