// sp_loop.cuh -- what the persistent cooperative kernels share: warp and block
// scans, the bounded grid barrier of the fixedPoint loops, and the test that
// lets a repair kernel run.
#pragma once

#include "sp_graph.cuh"

namespace sp {

namespace {

constexpr u32 kFull = 0xffffffffu;

__device__ __forceinline__ u32 warp_incl_scan(u32 x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    u32 y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
  return x;
}

__device__ __forceinline__ u64 shfl64(u64 x, int src) {
  u32 lo = __shfl_sync(kFull, (u32)x, src), hi = __shfl_sync(kFull, (u32)(x >> 32), src);
  return ((u64)hi << 32) | lo;
}
__device__ __forceinline__ u64 shfl64_down(u64 x, int d) {
  u32 lo = __shfl_down_sync(kFull, (u32)x, d), hi = __shfl_down_sync(kFull, (u32)(x >> 32), d);
  return ((u64)hi << 32) | lo;
}

// Grid barrier over a monotone arrival count: barrier k of a launch waits
// for k * gridDim.x arrivals (the count is zeroed at the start of every
// call).  Every wait is bounded by lim.wait_ns; a wait that runs out sets
// ctl->timeout = 2 and returns, and every later wait returns at once.
__device__ __forceinline__ u64 ld_acquire_u64(const u64 *p) {
  u64 v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

//
// Returns whether a timeout has been raised (the same answer in every thread
// of the block, so that loops leave in step and no __syncthreads is left
// waiting for threads that have gone).
// With `src`, thread 0 also reads the next round's frontier counters once
// the wait is over and hands them to the block in *out: one read per block
// instead of one per warp, all of them at the same line.
struct RoundCounts {
  u64 q;        // next frontier: entries << 32 | edges
  u32 ns;       // its small list
  u32 nf, fm;   // far pile: count and smallest distance (0, ~0 without one)
};
struct CountSrc {
  const u64 *q;
  const u32 *ns, *nf, *fm;   // nf, fm null without a far pile
};

__device__ __forceinline__ bool grid_sync(u64 *bar, u64 target, Ctl *c, const Limits &lim,
                                          const CountSrc *src = nullptr,
                                          RoundCounts *out = nullptr) {
  __shared__ int s_stop;
  __shared__ RoundCounts s_rc;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    // the count before this arrival says whether it was the last one; the
    // wait polls the count alone and looks at the timeout flag and the
    // clock every 16th poll (on every poll where the bound is that short)
    // (the test hook lim.miss_site == 2: block 0 does not arrive)
    const bool miss = lim.miss_site == 2u && blockIdx.x == 0;
    const u64 arrived = miss ? ld_acquire_u64(bar) : atomicAdd((unsigned long long *)bar, 1ull) + 1;
    if (arrived < target) {
      const u64 t0 = globaltimer_ns();
      u32 polls = 0;
      while (ld_acquire_u64(bar) < target) {
        if ((++polls & clock_polls(lim.wait_ns)) == 0) {
          if (ld_cg_i32(&c->timeout) != 0) break;
          if (globaltimer_ns() - t0 > lim.wait_ns || polls > kMaxPolls) {
            raise_timeout(c, 2, 2, (u32)(target / gridDim.x));
            break;
          }
        }
        __nanosleep(64);
      }
    }
    s_stop = ld_cg_i32(&c->timeout) != 0;
    if (src) {
      s_rc.q = ld_cg_u64(src->q);
      s_rc.ns = ld_cg_u32(src->ns);
      s_rc.nf = src->nf ? ld_cg_u32(src->nf) : 0u;
      s_rc.fm = src->fm ? ld_cg_u32(src->fm) : 0xFFFFFFFFu;
    }
  }
  __syncthreads();
  if (src) *out = s_rc;
  return s_stop != 0;
}

// Block scan helper: exclusive prefix of one value per thread; the block
// total goes to *total (smem scratch of 33 words).
__device__ __forceinline__ u32 block_excl_scan(u32 x, u32 *scratch, u32 *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const u32 incl = warp_incl_scan(x);
  if (lane == 31) scratch[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    u32 v = lane < nwarps ? scratch[lane] : 0u;
    v = warp_incl_scan(v);
    if (lane < nwarps) scratch[lane] = v;
  }
  __syncthreads();
  const u32 r = (warp ? scratch[warp - 1] : 0u) + incl - x;
  *total = scratch[nwarps - 1];
  __syncthreads();
  return r;
}

// (one 16-byte read and one more beside it, not four one after the other)
__device__ __forceinline__ bool repair_enabled(Ctl *c) {
  const int4 f = __ldcg((const int4 *)&c->status);   // status, need_grow, range_err, timeout
  return (f.x | f.y | f.w | ld_cg_i32(&c->bad)) == 0;
}

// The same test with one answer for the whole block (kernels with barriers).
__device__ __forceinline__ bool repair_enabled_block(Ctl *c) {
  __shared__ int s_ok;
  if (threadIdx.x == 0) s_ok = repair_enabled(c) ? 1 : 0;
  __syncthreads();
  return s_ok != 0;
}

// The end of a call in the kernel that ends it (block-collective, every block
// of the grid): the last block to get here does the call's bookkeeping and
// writes the control block into the host's pinned copy, as k_finish does, but
// without a launch of its own (a call with 64 updates: 5 of 112 us).
__device__ __forceinline__ void finish_call(Ctl *c, Ctl *host) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(&c->done, 1u) == gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  if (!s_last) return;
  if (threadIdx.x == 0 && ld_cg_i32(&c->status) == 0 && ld_cg_i32(&c->need_grow) == 0) {
    c->pool_used[0] = ld_cg_u64(&c->pool_need[0]);
    c->pool_used[1] = ld_cg_u64(&c->pool_need[1]);
  }
  __syncthreads();
  const u32 *src = (const u32 *)c;
  u32 *dst = (u32 *)host;
  for (u32 i = threadIdx.x; i < sizeof(Ctl) / 4; i += blockDim.x) dst[i] = __ldcg(src + i);
}

}  // namespace

}  // namespace sp
