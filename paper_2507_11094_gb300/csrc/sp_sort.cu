// sp_sort.cu -- stable LSD radix sort of (u64 key, u32 value) pairs.
//
// Groups a batch's updates by (store, row, col) so that each touched row is
// merged once (updateCSRDel / updateCSRAdd of the DynSSSP driver, done as a
// sort-merge), and orders graph edges when a store is built.
//
// The edge sort, per digit of at most 8 bits, over tiles of 4,096 pairs:
//   k_hist       a tile's digit counts (the count table is digit-major);
//   k_digit_scan one block per digit: prefix of its counts over the tiles,
//                and the digit's total;
//   k_scatter    digit bases from the totals, a stable rank of the tile's
//                pairs (ballots per digit bit, warp-private digit counters),
//                the pairs staged in shared memory in digit order, and runs of
//                a digit written out by consecutive threads.
// What bounds a pass is its 24 bytes per pair of reads and writes, if the runs
// are long enough to fill sectors: a tile of 4,096 has 16 or more pairs per
// digit.  16.8 M pairs (R-MAT 20's reverse store, three 7-bit passes because
// the input is in row order already): 2.3 -> 0.43 ms, a scatter 190-470 ->
// 110 us (3.6 TB/s), against five passes over tiles of 1,024 pairs with 512
// bins: two pairs a run, the next digit counted by 16.8 M global atomics a
// pass and a count table of 33 MB.
#include "sp_graph.cuh"

#include <algorithm>
#include <type_traits>

namespace sp {

namespace {

constexpr int kBinsMax = 1 << 10;       // digits of the batch sort: 9 or 10 bits
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxDigit = 8;           // digits of the edge sort
constexpr int kSBins = 1 << kMaxDigit;
constexpr int kST = 512;               // its threads per block,
constexpr int kSW = kST / 32;
constexpr int kSItems = 8;             // pairs per thread
constexpr int kSTile = kST * kSItems;  // and pairs per tile

__global__ void __launch_bounds__(kST)
k_hist(const u64 *__restrict__ keys, long long n, int shift, int bins, u32 *__restrict__ counts,
       u32 tiles) {
  __shared__ u32 h[kSBins];
  if (threadIdx.x < kSBins) h[threadIdx.x] = 0;
  __syncthreads();
  const long long base = (long long)blockIdx.x * kSTile;
  u32 d[kSItems];
#pragma unroll
  for (int k = 0; k < kSItems; ++k) {   // all loads first, then the counts
    const long long i = base + k * kST + threadIdx.x;
    d[k] = i < n ? (u32)(keys[i] >> shift) & (u32)(bins - 1) : 0xFFFFFFFFu;
  }
#pragma unroll
  for (int k = 0; k < kSItems; ++k)
    if (d[k] != 0xFFFFFFFFu) atomicAdd(&h[d[k]], 1u);
  __syncthreads();
  if ((int)threadIdx.x < bins) counts[(long long)threadIdx.x * tiles + blockIdx.x] = h[threadIdx.x];
}

__device__ __forceinline__ u32 warp_incl_scan(u32 x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u32 y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// Block-wide exclusive scan of one value per thread (256 threads).
__device__ __forceinline__ u32 block_excl_scan(u32 x, u32 *ws, u32 *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u32 incl = warp_incl_scan(x);
  if (lane == 31) ws[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    u32 v = lane < kWarps ? ws[lane] : 0u;
    v = warp_incl_scan(v);
    if (lane < kWarps) ws[lane] = v;
  }
  __syncthreads();
  const u32 r = (warp ? ws[warp - 1] : 0u) + incl - x;
  *total = ws[kWarps - 1];
  __syncthreads();
  return r;
}

// Block d: exclusive prefix of counts[d][0..tiles) in place, total to
// totals[d].
__global__ void __launch_bounds__(kThreads)
k_digit_scan(u32 *__restrict__ counts, u32 tiles, u32 *__restrict__ totals) {
  __shared__ u32 ws[kWarps];
  u32 *row = counts + (long long)blockIdx.x * tiles;
  const u32 per = (tiles + kThreads - 1) / kThreads;
  const u32 b = threadIdx.x * per < tiles ? threadIdx.x * per : tiles;
  const u32 e = b + per < tiles ? b + per : tiles;
  u32 sum = 0;
  for (u32 i = b; i < e; ++i) sum += row[i];
  u32 total;
  u32 run = block_excl_scan(sum, ws, &total);
  for (u32 i = b; i < e; ++i) {
    const u32 x = row[i];
    row[i] = run;
    run += x;
  }
  if (threadIdx.x == 0) totals[blockIdx.x] = total;
}

// Block-wide exclusive scan over 512 threads.
__device__ __forceinline__ u32 bscan512(u32 x, u32 *ws, u32 *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u32 incl = warp_incl_scan(x);
  if (lane == 31) ws[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    u32 v = lane < kSW ? ws[lane] : 0u;
    v = warp_incl_scan(v);
    if (lane < kSW) ws[lane] = v;
  }
  __syncthreads();
  const u32 r = (warp ? ws[warp - 1] : 0u) + incl - x;
  *total = ws[kSW - 1];
  __syncthreads();
  return r;
}

// Lanes of the warp whose valid item has the same kB-bit digit (the answer of
// a match_any, built from one ballot per digit bit).
template <int kB>
__device__ __forceinline__ u32 digit_peers(u32 d, bool valid) {
  u32 peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
  for (int bb = 0; bb < kB; ++bb) {
    const bool on = (d >> bb) & 1;
    const u32 bal = __ballot_sync(0xffffffffu, on);
    peers &= on ? bal : ~bal;
  }
  return peers;
}

constexpr size_t kSSmem = (size_t)kSTile * (sizeof(u64) + sizeof(u32));

__global__ void __launch_bounds__(kST, 2)
k_scatter(const u64 *__restrict__ keys, const u32 *__restrict__ vals, long long n, int shift,
          int bins, const u32 *__restrict__ offs, const u32 *__restrict__ totals, u32 tiles,
          u64 *__restrict__ keys_out, u32 *__restrict__ vals_out) {
  extern __shared__ __align__(16) unsigned char smraw[];
  u64 *s_key = (u64 *)smraw;                  // [kSTile]
  u32 *s_val = (u32 *)(s_key + kSTile);       // [kSTile]
  __shared__ u32 s_wc[kSW][kSBins];           // digit counts of each warp, then its offsets
  __shared__ u32 s_off[kSBins];               // where the tile's run of a digit goes, less its
                                              // place in the tile
  __shared__ u32 ws[kSW];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const long long base = (long long)blockIdx.x * kSTile;
  const u32 left = (u32)(n - base < kSTile ? n - base : kSTile);
  const u32 w0 = (u32)warp * (32 * kSItems);
  u64 rk[kSItems];
  u32 rv[kSItems], lr[kSItems];
#pragma unroll
  for (int k = 0; k < kSItems; ++k) {   // the whole tile is in flight at once
    const u32 i = w0 + k * 32 + lane;
    rk[k] = i < left ? __ldcs(keys + base + i) : 0ull;
    rv[k] = i < left ? __ldcs(vals + base + i) : 0u;
  }
#pragma unroll
  for (int w = 0; w < kSW * kSBins / kST; ++w) ((u32 *)s_wc)[w * kST + t] = 0;
  u32 tot_d = 0, off_d = 0;
  if (t < bins) {
    tot_d = totals[t];
    off_d = offs[(long long)t * tiles + blockIdx.x];
  }
  u32 all;
  off_d += bscan512(tot_d, ws, &all);   // (its barriers order the clearing, too)
  // stable rank within the warp's pairs (rows k, then lanes)
  const u32 lt = lanemask_lt();
  u32 *wc = s_wc[warp];
#pragma unroll
  for (int k = 0; k < kSItems; ++k) {
    const bool valid = w0 + k * 32 + lane < left;
    const u32 d = (u32)(rk[k] >> shift) & (u32)(bins - 1);
    const u32 peers = digit_peers<kMaxDigit>(d, valid);
    const u32 rank = __popc(peers & lt);
    const u32 before = valid ? wc[d] : 0u;
    __syncwarp();
    if (valid && rank == 0) wc[d] = before + __popc(peers);
    __syncwarp();
    lr[k] = before + rank;
  }
  __syncthreads();
  {   // digit t: offsets of the warps, then of the digit in the tile
    u32 run = 0;
    if (t < kSBins) {
#pragma unroll
      for (int w = 0; w < kSW; ++w) {
        const u32 x = s_wc[w][t];
        s_wc[w][t] = run;
        run += x;
      }
    }
    const u32 loc = bscan512(run, ws, &all);
    if (t < kSBins) {
#pragma unroll
      for (int w = 0; w < kSW; ++w) s_wc[w][t] += loc;
      s_off[t] = off_d - loc;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kSItems; ++k) {
    if (w0 + k * 32 + lane < left) {
      const u32 d = (u32)(rk[k] >> shift) & (u32)(bins - 1);
      const u32 lp = wc[d] + lr[k];
      s_key[lp] = rk[k];
      s_val[lp] = rv[k];
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kSItems; ++k) {
    const u32 j = k * kST + t;
    if (j < left) {
      const u64 key = s_key[j];
      const u32 pos = s_off[(u32)(key >> shift) & (u32)(bins - 1)] + j;
      keys_out[pos] = key;
      vals_out[pos] = s_val[j];
    }
  }
}

// ---------------------------------------------------------------------------
// The batch sort: one cooperative launch builds the items of a batch, sorts
// them by (store, row, col, kind) and emits one segment per touched
// (store, row) -- the grouping that lets every touched row be merged once
// (updateCSRDel + updateCSRAdd of the DynSSSP driver as one sort-merge).
//
// Block b owns a contiguous chunk of item positions.  Items arrive forward
// store first and, within a store, deletions first, and every pass is stable:
// so the kind bit is never sorted on, and where the grid has two blocks or
// more, half of them sorts the forward items and half the reverse ones, each
// within its own half of the positions, and the store's bit is not sorted on
// either.  That leaves 2 * bits key bits, in digits of ten bits where this
// saves a pass over nine (ids of 5, 10, 14, 15, 19, 20, 23 to 25 and 28 to 30
// bits): on R-MAT 20 four passes instead of five, on R-MAT 22 five (nine bits) instead of six.  A pass
// is two grid barriers, a scatter and a read back.  A batch and its undo of
// 1,000,000 updates on R-MAT 22: 2,398 -> 2,369 us, of 161,000 on 32 graphs
// together: 1,070 -> 1,058 us, of 20,971 pairs in the triangle count: 1,012 ->
// 987 us; R-MAT 20 and 167,772 updates: 816 us either way (the searches beside
// the sort take as long).  A batch within one tile is sorted by one block with
// the store's bit.  Per pass:
//   1. the block counts the digit over its chunk and writes the counts as
//      row b of a table (chunk-major);                     -- grid barrier
//   2. the threads read the table's columns (coalesced across the warp): a
//      digit's total and its count in earlier chunks of its half; a block scan of the totals
//      gives the digit bases;
//   3. per sub-tile of kBTile items (warp w holds items w*256 .. w*256+255,
//      eight per lane): each warp ranks its items with match_any against
//      warp-private digit counters, one scan over the warps per digit
//      turns those into offsets, the items are staged in shared memory in
//      digit order and written out so that consecutive threads store
//      consecutive positions of a digit's run.             -- grid barrier
// A chunk of one sub-tile keeps its items in registers from the count to
// the scatter.  Data other blocks wrote is read through L2 (.cg), and
// loads are issued in unrolled batches so that their latencies overlap.
// ---------------------------------------------------------------------------
constexpr int kBT = 512;                  // threads per block (one or two digits each)
constexpr int kBW = kBT / 32;
constexpr int kBItems = 8;
constexpr int kBTile = kBT * kBItems;     // items per sub-tile
constexpr int kBWarpItems = 32 * kBItems; // items per warp and sub-tile
static_assert(kBT == kST, "bscan512");
// dynamic shared memory: staged keys and values, per-warp digit counters,
// four per-digit arrays
template <int KB>
constexpr size_t kBSmem = (size_t)kBTile * (sizeof(u64) + sizeof(u32)) +
                          (size_t)(kBW * kBT + 4 * (1 << KB)) * 4;

struct BatchSortArgs {
  const int *ds, *dd, *as, *ad, *aw;
  long long nd, na;
  int n, bits, passes;
  u64 *kbuf[2];
  u32 *vbuf[2];
  u32 *tab;          // [G][1 << KB] digit counts per chunk
  Seg *seg;
  Ctl *ctl;
  unsigned long long wait_ns;
  u32 miss_site;         // test hook of the bounded waits (Limits::miss_site)
  u32 n_items, chunk;
  u32 halves;        // 2: half of the grid per store
};

__device__ __forceinline__ u64 shfl64_up1(u64 x) {
  const u32 lo = __shfl_up_sync(0xffffffffu, (u32)x, 1);
  const u32 hi = __shfl_up_sync(0xffffffffu, (u32)(x >> 32), 1);
  return ((u64)hi << 32) | lo;
}

// Position of item k of this thread in its sub-tile.
__device__ __forceinline__ u32 sub_pos(int k) {
  return (threadIdx.x >> 5) * kBWarpItems + k * 32 + (threadIdx.x & 31);
}

// KB bits a digit.  Per-warp digit counters: 32-bit at nine bits, pairs of 16
// bits at ten (a sub-tile has 4,096 items), so 512 words a warp either way.
template <int KB>
__global__ void __launch_bounds__(kBT) k_batch_sort(BatchSortArgs a) {
  constexpr int kBins = 1 << KB, kDT = kBins / kBT;   // digits, and digits per thread
  static_assert(kDT == 1 || kDT == 2, "counter words");
  using Cnt = std::conditional_t<kDT == 1, u32, unsigned short>;
  extern __shared__ __align__(16) unsigned char smraw[];
  u64 *s_key = (u64 *)smraw;                         // [kBTile]
  u32 *s_val = (u32 *)(s_key + kBTile);              // [kBTile]
  u32 *s_wc = s_val + kBTile;                        // [kBW][kBT] words of per-warp digit counts
  u32 *s_off = s_wc + kBW * kBT;                   // global start of digit (next sub-tile)
  u32 *s_run = s_off + kBins;
  u32 *s_loc = s_run + kBins;                        // sub-tile start of digit
  u32 *s_hist = s_loc + kBins;                       // digit counts
  __shared__ u32 ws[kBW];
  Ctl *c = a.ctl;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const u32 G = gridDim.x, b = blockIdx.x;
  // this block's half of the grid and of the positions, and its chunk there
  const u32 Gh = G / a.halves, half = b / Gh, bh = b - half * Gh;
  const u32 nh0 = half * (a.n_items / a.halves), nh1 = nh0 + a.n_items / a.halves;
  const u32 cb = min(nh0 + bh * a.chunk, nh1), ce = min(cb + a.chunk, nh1);
  const bool one = ce - cb <= (u32)kBTile;           // the chunk is one sub-tile
  u64 *bar = &c->bar_sort;
  u64 nbar = 0;
  const long long nb = a.nd + a.na;
  const int bits = a.bits;
  const u32 lt = lanemask_lt();
  u64 rk[kBItems];
  u32 rv[kBItems];

  // the items (forward item of update i at i, reverse item at nb + i; the
  // low key bit is 0 for a deletion and 1 for an insertion, so a deletion
  // sorts before an insertion of the same edge) with the first digit's
  // counts; an invalid id or weight raises SP_EINVAL (nothing will change)
#pragma unroll
  for (int e = 0; e < kDT; ++e) s_hist[e * kBT + t] = 0;
  __syncthreads();
  for (u32 tb = cb; tb < ce; tb += kBTile) {
    int u[kBItems], v[kBItems], w[kBItems];
#pragma unroll
    for (int k = 0; k < kBItems; ++k) {   // every load first
      const u32 i = tb + sub_pos(k);
      u[k] = 0; v[k] = 0; w[k] = 0;
      if (i < ce) {
        const long long j = (long long)i >= nb ? (long long)i - nb : (long long)i;
        if (j < a.nd) {
          u[k] = __ldg(a.ds + j); v[k] = __ldg(a.dd + j); w[k] = 0;
        } else {
          const long long q = j - a.nd;
          u[k] = __ldg(a.as + q); v[k] = __ldg(a.ad + q); w[k] = __ldg(a.aw + q);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < kBItems; ++k) {
      const u32 i = tb + sub_pos(k);
      rk[k] = 0;
      rv[k] = 0;
      if (i < ce) {
        const bool rev = (long long)i >= nb;
        const long long j = rev ? (long long)i - nb : (long long)i;
        const u64 kind = j < a.nd ? 0 : 1;
        const bool ok = u[k] >= 0 && u[k] < a.n && v[k] >= 0 && v[k] < a.n &&
                        (kind == 0 || (w[k] >= 1 && w[k] <= SP_WMAX));
        if (!ok) {
          atomicCAS(&c->status, 0, SP_EINVAL);
          u[k] = 0; v[k] = 0;
        }
        rk[k] = rev ? (1ull << (2 * bits + 1)) | ((u64)v[k] << (bits + 1)) | ((u64)u[k] << 1) | kind
                    : ((u64)u[k] << (bits + 1)) | ((u64)v[k] << 1) | kind;
        rv[k] = i;   // the item's own number: its search result and weight (k_search)
      }
    }
#pragma unroll
    for (int k = 0; k < kBItems; ++k) {
      const u32 i = tb + sub_pos(k);
      if (i < ce) {
        a.kbuf[0][i] = rk[k];
        a.vbuf[0][i] = rv[k];
        atomicAdd(&s_hist[(rk[k] >> 1) & (kBins - 1)], 1u);
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < kDT; ++e) a.tab[(size_t)b * kBins + e * kBT + t] = s_hist[e * kBT + t];

  for (int p = 0; p < a.passes; ++p) {
    if (coop_barrier(bar, ++nbar * G, c, a.wait_ns, 4, a.miss_site)) return;
    const int shift = 1 + p * KB;   // above the kind bit
    // digit bases of this chunk: thread t sums digits 4*(t % kPer) .. +3 over
    // its half's rows q = t / kPer (mod kRows) with 16-byte loads; the partial
    // sums of each digit meet in shared memory (s_loc holds the totals, s_run
    // the counts of earlier chunks)
    {
      constexpr u32 kPer = kBins / 4, kRows = kBT / kPer;
      const u32 *tab = a.tab + (size_t)half * Gh * kBins;
      const u32 dq = ((u32)t & (kPer - 1)) * 4, rg = (u32)t / kPer;
      uint4 tot = make_uint4(0u, 0u, 0u, 0u), pre = tot;
      for (u32 q0 = rg; q0 < Gh; q0 += kRows * 8) {
        uint4 x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const u32 q = q0 + kRows * u;
          x[u] = q < Gh ? __ldcg((const uint4 *)(tab + (size_t)q * kBins + dq))
                        : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const bool before = q0 + kRows * u < bh;
          tot.x += x[u].x; tot.y += x[u].y; tot.z += x[u].z; tot.w += x[u].w;
          if (before) { pre.x += x[u].x; pre.y += x[u].y; pre.z += x[u].z; pre.w += x[u].w; }
        }
      }
#pragma unroll
      for (int e = 0; e < kDT; ++e) {
        s_loc[e * kBT + t] = 0;
        s_run[e * kBT + t] = 0;
      }
      __syncthreads();
      atomicAdd(&s_loc[dq], tot.x); atomicAdd(&s_loc[dq + 1], tot.y);
      atomicAdd(&s_loc[dq + 2], tot.z); atomicAdd(&s_loc[dq + 3], tot.w);
      atomicAdd(&s_run[dq], pre.x); atomicAdd(&s_run[dq + 1], pre.y);
      atomicAdd(&s_run[dq + 2], pre.z); atomicAdd(&s_run[dq + 3], pre.w);
      __syncthreads();
      u32 all, mine = 0;
#pragma unroll
      for (int e = 0; e < kDT; ++e) mine += s_loc[t * kDT + e];
      u32 base = nh0 + bscan512(mine, ws, &all);
#pragma unroll
      for (int e = 0; e < kDT; ++e) {
        s_off[t * kDT + e] = base + s_run[t * kDT + e];
        base += s_loc[t * kDT + e];
      }
    }
    const u64 *kin = a.kbuf[p & 1];
    const u32 *vin = a.vbuf[p & 1];
    u64 *kout = a.kbuf[(p + 1) & 1];
    u32 *vout = a.vbuf[(p + 1) & 1];
    for (u32 tb = cb; tb < ce; tb += kBTile) {
      if (!one) {   // this sub-tile's items and digit counts
#pragma unroll
        for (int k = 0; k < kBItems; ++k) {
          const u32 i = tb + sub_pos(k);
          rk[k] = i < ce ? __ldcg(kin + i) : 0ull;
          rv[k] = i < ce ? __ldcg(vin + i) : 0u;
        }
#pragma unroll
        for (int e = 0; e < kDT; ++e) s_hist[e * kBT + t] = 0;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kBItems; ++k)
          if (tb + sub_pos(k) < ce) atomicAdd(&s_hist[(rk[k] >> shift) & (kBins - 1)], 1u);
        __syncthreads();
      }
      {
        u32 all, mine = 0;
#pragma unroll
        for (int e = 0; e < kDT; ++e) mine += s_hist[t * kDT + e];
        u32 base = bscan512(mine, ws, &all);
#pragma unroll
        for (int e = 0; e < kDT; ++e) {
          s_loc[t * kDT + e] = base;
          base += s_hist[t * kDT + e];
        }
#pragma unroll
        for (int w = 0; w < kBW; ++w) s_wc[w * kBT + t] = 0;
      }
      __syncthreads();
      // stable rank within the warp's items (rows k, then lanes)
      u32 lr[kBItems];
      Cnt *wc = (Cnt *)(s_wc + warp * kBT);
#pragma unroll
      for (int k = 0; k < kBItems; ++k) {
        const bool valid = tb + sub_pos(k) < ce;
        const u32 d = (u32)((rk[k] >> shift) & (kBins - 1));
        const u32 peers = digit_peers<KB>(d, valid);
        const u32 rank = __popc(peers & lt);
        const u32 before = valid ? (u32)wc[d] : 0u;
        __syncwarp();
        if (valid && rank == 0) wc[d] = (Cnt)(before + __popc(peers));
        __syncwarp();
        lr[k] = before + rank;
      }
      __syncthreads();
      {   // word t (a digit, or two of 16 bits): offsets of the warps
        u32 run = 0;
#pragma unroll
        for (int w = 0; w < kBW; ++w) {
          const u32 x = s_wc[w * kBT + t];
          s_wc[w * kBT + t] = run;
          run += x;
        }
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < kBItems; ++k) {
        if (tb + sub_pos(k) < ce) {
          const u32 d = (u32)((rk[k] >> shift) & (kBins - 1));
          const u32 lp = s_loc[d] + wc[d] + lr[k];
          s_key[lp] = rk[k];
          s_val[lp] = rv[k];
        }
      }
      __syncthreads();
      // write out in digit order: a digit's items are consecutive in both
#pragma unroll
      for (int k = 0; k < kBItems; ++k) {
        const u32 j = k * kBT + t;
        if (tb + j < ce) {
          const u64 key = s_key[j];
          const u32 d = (u32)((key >> shift) & (kBins - 1));
          const u32 pos = s_off[d] + (j - s_loc[d]);
          kout[pos] = key;
          vout[pos] = s_val[j];
        }
      }
      __syncthreads();
#pragma unroll
      for (int e = 0; e < kDT; ++e) s_off[e * kBT + t] += s_hist[e * kBT + t];
      __syncthreads();
    }
    if (coop_barrier(bar, ++nbar * G, c, a.wait_ns, 4, a.miss_site)) return;
    if (p + 1 < a.passes) {   // the next digit's counts over this chunk
      const int nshift = shift + KB;
#pragma unroll
      for (int e = 0; e < kDT; ++e) s_hist[e * kBT + t] = 0;
      __syncthreads();
      for (u32 tb = cb; tb < ce; tb += kBTile) {
#pragma unroll
        for (int k = 0; k < kBItems; ++k) {
          const u32 i = tb + sub_pos(k);
          rk[k] = i < ce ? __ldcg(kout + i) : 0ull;
          if (one) rv[k] = i < ce ? __ldcg(vout + i) : 0u;
        }
#pragma unroll
        for (int k = 0; k < kBItems; ++k)
          if (tb + sub_pos(k) < ce) atomicAdd(&s_hist[(rk[k] >> nshift) & (kBins - 1)], 1u);
      }
      __syncthreads();
#pragma unroll
      for (int e = 0; e < kDT; ++e) a.tab[(size_t)b * kBins + e * kBT + t] = s_hist[e * kBT + t];
    }
  }

  // segments: a head is an item whose (store, row) differs from its
  // predecessor's.  Items sit as in the passes (warp w, row k, lane), so a
  // predecessor is one lane back (or the previous row's last lane); heads
  // become ballot masks, a segment ends at the next head -- in the same
  // row, a later row, a later warp of the block (a minimum over the warps),
  // or, only for a row of the graph that runs past the sub-tile, where a
  // galloping search finds it.
  const u64 *keys = a.kbuf[a.passes & 1];
  const u32 n = a.n_items;
  const int hs = bits + 1;
  for (u32 tb = cb; tb < ce; tb += kBTile) {
    const u32 te = tb + kBTile < ce ? tb + kBTile : ce;
    u64 pf[kBItems];
    u32 hm[kBItems];
#pragma unroll
    for (int k = 0; k < kBItems; ++k) {
      const u32 i = tb + sub_pos(k);
      pf[k] = i < te ? __ldcg(keys + i) >> hs : 0ull;
    }
    const u32 w0 = tb + (u32)warp * kBWarpItems;   // the warp's first position
    const u64 before0 = (w0 > 0 && w0 < te) ? __ldcg(keys + w0 - 1) >> hs : ~0ull;
    u32 nh = 0;
#pragma unroll
    for (int k = 0; k < kBItems; ++k) {
      const u32 i = tb + sub_pos(k);
      u64 pred = shfl64_up1(pf[k]);
      const u64 last_prev = __shfl_sync(0xffffffffu, (u32)(k ? pf[k - 1] : before0), 31) |
                            ((u64)__shfl_sync(0xffffffffu, (u32)((k ? pf[k - 1] : before0) >> 32), 31) << 32);
      if (lane == 0) pred = k ? last_prev : before0;
      const bool head = i < te && (i == 0 || pf[k] != pred);
      hm[k] = __ballot_sync(0xffffffffu, head);
      nh += __popc(hm[k]);
    }
    // the warp's first head, its head count, then the block's prefix
    u32 first = 0xFFFFFFFFu;
#pragma unroll
    for (int k = kBItems - 1; k >= 0; --k)
      if (hm[k]) first = w0 + (u32)k * 32 + (u32)(__ffs(hm[k]) - 1);
    if (lane == 0) {
      s_hist[warp] = nh;
      s_loc[warp] = first;
    }
    __syncthreads();
    if (t == 0) {
      u32 tot = 0;
      for (int w = 0; w < kBW; ++w) {
        const u32 x = s_hist[w];
        s_hist[w] = tot;
        tot += x;
      }
      s_run[0] = tot ? atomicAdd(&c->n_seg, tot) : 0u;
    }
    u32 after = 0xFFFFFFFFu;   // first head of a later warp
    for (int w = warp + 1; w < kBW; ++w) after = min(after, s_loc[w]);
    __syncthreads();
    u32 sidx = s_run[0] + s_hist[warp];
#pragma unroll
    for (int k = 0; k < kBItems; ++k) {
      const u32 mine = hm[k] & lt;
      if ((hm[k] >> lane) & 1) {
        const u32 i = tb + sub_pos(k);
        const u64 pfx = pf[k];
        u32 end = 0xFFFFFFFFu;
        const u32 above = hm[k] & ~((2u << lane) - 1);   // later heads in this row
        if (above) {
          end = w0 + (u32)k * 32 + (u32)(__ffs(above) - 1);
        } else {
#pragma unroll
          for (int k2 = k + 1; k2 < kBItems; ++k2)
            if (end == 0xFFFFFFFFu && hm[k2]) end = w0 + (u32)k2 * 32 + (u32)(__ffs(hm[k2]) - 1);
        }
        if (end == 0xFFFFFFFFu) end = after;
        if (end == 0xFFFFFFFFu) {   // the row runs past the sub-tile
          u32 lo = te, step = 1;
          u32 hi = lo;
          while (hi < n && (__ldcg(keys + hi) >> hs) == pfx) {
            lo = hi + 1;
            hi = lo + step < n ? lo + step : n;
            step <<= 1;
          }
          while (lo < hi) {   // first item of another (store, row) in [lo, hi]
            const u32 mid = (lo + hi) >> 1;
            if ((__ldcg(keys + mid) >> hs) == pfx) lo = mid + 1; else hi = mid;
          }
          end = lo;
        }
        Seg &sg = a.seg[sidx + __popc(mine)];
        sg.first = i;
        sg.end = end;
        sg.row = (int)(pfx & ((1ull << bits) - 1));
        sg.dir = (int)(pfx >> bits);
      }
      sidx += __popc(hm[k]);
    }
    __syncthreads();
  }
}

}  // namespace

size_t sort_tmp_bytes(long long n) {
  const long long tiles = (n + kSTile - 1) / kSTile;
  return (size_t)(tiles * kSBins + kSBins + 64) * sizeof(u32) + 256;
}

// Co-resident blocks per SM of one digit width; 0 if it cannot run.
template <int KB>
static int sort_per_sm() {
  int per_sm = 0;
  if (cudaFuncSetAttribute(k_batch_sort<KB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)std::max(kBSmem<KB>, kExclusiveSmem)) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batch_sort<KB>, kBT, kBSmem<KB>) !=
          cudaSuccess)
    return 0;
  return per_sm;
}

int batch_sort_blocks(int num_sms) {
  return std::max(0, std::min(sort_per_sm<9>(), sort_per_sm<10>())) * num_sms;
}

size_t batch_sort_tmp_bytes(int max_blocks) {
  return (size_t)kBinsMax * std::max(max_blocks, 1) * sizeof(u32) + 256;
}

namespace {

// One launch of the batch sort: its kernel and dynamic shared memory.
struct SortLaunch {
  void (*fn)(BatchSortArgs);
  size_t smem;
  int G;
};

// How ni items are sorted: in one half or two, and the digits.
struct SortShape {
  int halves, passes;
  bool wide;   // ten bits a digit
};

SortShape sort_shape(const sp_graph *g, long long ni) {
  int cap = g->sort_blocks;
  if (g->loop_blocks_user > 0 && g->loop_blocks_user < cap) cap = g->loop_blocks_user;
  SortShape s;
  // two blocks or more: as many for either store
  s.halves = ni > kBTile && cap >= 2 ? 2 : 1;
  const int key_bits = 2 * g->bits + (s.halves == 1 ? 1 : 0);
  const int p9 = std::max((key_bits + 8) / 9, 1), p10 = std::max((key_bits + 9) / 10, 1);
  s.wide = p10 < p9;
  s.passes = s.wide ? p10 : p9;
  return s;
}

// Arguments and grid of the batch sort for these inputs.
SortLaunch batch_sort_args(sp_graph *g, const int *ds, const int *dd, long long nd,
                           const int *as, const int *ad, const int *aw, long long na,
                           BatchSortArgs &a) {
  const long long ni = 2 * (nd + na);
  BatchBufs &bb = g->bb;
  int cap = g->sort_blocks;
  if (g->loop_blocks_user > 0 && g->loop_blocks_user < cap) cap = g->loop_blocks_user;
  const SortShape sh = sort_shape(g, ni);
  a.halves = sh.halves;
  const long long nh = ni / (int)a.halves;
  const int Gh = (int)std::max(1ll, std::min<long long>((nh + kBTile - 1) / kBTile,
                                                        cap / (int)a.halves));
  const int G = Gh * (int)a.halves;
  a.ds = ds; a.dd = dd; a.as = as; a.ad = ad; a.aw = aw;
  a.nd = nd; a.na = na;
  a.n = g->n;
  a.bits = g->bits;
  a.passes = sh.passes;
  // the last pass writes keys/vals
  const int odd = a.passes & 1;
  a.kbuf[0] = odd ? bb.keys_alt : bb.keys;
  a.kbuf[1] = odd ? bb.keys : bb.keys_alt;
  a.vbuf[0] = odd ? bb.vals_alt : bb.vals;
  a.vbuf[1] = odd ? bb.vals : bb.vals_alt;
  a.tab = (u32 *)bb.tmp;
  a.seg = bb.seg;
  a.ctl = g->ctl;
  a.wait_ns = g->lim.wait_ns;
  a.miss_site = g->lim.miss_site;
  a.n_items = (u32)ni;
  a.chunk = (u32)((nh + Gh - 1) / Gh);
  // a handle with a block share gives each block an SM of its own
  const size_t least = g->loop_blocks_user > 0 ? kExclusiveSmem : 0;
  if (sh.wide) return {k_batch_sort<10>, std::max(kBSmem<10>, least), G};
  return {k_batch_sort<9>, std::max(kBSmem<9>, least), G};
}

}  // namespace

int batch_sort_passes(const sp_graph *g, long long ni) { return sort_shape(g, ni).passes; }

bool is_batch_sort(const void *fn) {
  return fn == (const void *)k_batch_sort<9> || fn == (const void *)k_batch_sort<10>;
}

cudaError_t launch_batch_sort(sp_graph *g, const int *ds, const int *dd, long long nd,
                              const int *as, const int *ad, const int *aw, long long na,
                              int *launches) {
  if (nd + na == 0) return cudaSuccess;
  BatchSortArgs a;
  const SortLaunch l = batch_sort_args(g, ds, dd, nd, as, ad, aw, na, a);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)l.G);
  cfg.blockDim = dim3(kBT);
  cfg.dynamicSmemBytes = l.smem;
  cfg.stream = g->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;   // all blocks co-resident
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  ++*launches;
  return cudaLaunchKernelEx(&cfg, l.fn, a);
}

cudaError_t retarget_batch_sort(sp_graph *g, cudaGraphExec_t ex, cudaGraphNode_t node,
                                const int *ds, const int *dd, long long nd, const int *as,
                                const int *ad, const int *aw, long long na) {
  BatchSortArgs a;
  const SortLaunch l = batch_sort_args(g, ds, dd, nd, as, ad, aw, na, a);
  void *args[1] = {&a};
  cudaKernelNodeParams p = {};
  p.func = (void *)l.fn;
  p.gridDim = dim3((unsigned)l.G);
  p.blockDim = dim3(kBT);
  p.sharedMemBytes = (unsigned)l.smem;
  p.kernelParams = args;
  return cudaGraphExecKernelNodeSetParams(ex, node, &p);
}

bool sort_pairs(u64 *keys, u32 *vals, u64 *keys_alt, u32 *vals_alt, long long n, int lo_bit,
                int hi_bit, void *tmp, cudaStream_t st, int *launches) {
  const int bits = hi_bit - lo_bit;
  if (n <= 1 || bits <= 0) return false;
  const u32 tiles = (u32)((n + kSTile - 1) / kSTile);
  u32 *counts = (u32 *)tmp;
  u32 *totals = counts + (long long)tiles * kSBins;
  u64 *kin = keys, *kout = keys_alt;
  u32 *vin = vals, *vout = vals_alt;
  // as few passes as kMaxDigit allows, of equal digits
  const int passes = (bits + kMaxDigit - 1) / kMaxDigit;
  const int digit = (bits + passes - 1) / passes;
  cudaFuncSetAttribute(k_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSSmem);
  for (int shift = lo_bit; shift < hi_bit; shift += digit) {
    const int bins = 1 << std::min(digit, hi_bit - shift);
    k_hist<<<tiles, kST, 0, st>>>(kin, n, shift, bins, counts, tiles);
    k_digit_scan<<<bins, kThreads, 0, st>>>(counts, tiles, totals);
    k_scatter<<<tiles, kST, kSSmem, st>>>(kin, vin, n, shift, bins, counts, totals, tiles, kout,
                                          vout);
    if (launches) *launches += 3;
    std::swap(kin, kout);
    std::swap(vin, vout);
  }
  return kin != keys;
}

}  // namespace sp
