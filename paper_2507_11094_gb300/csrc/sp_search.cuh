// sp_search.cuh -- searching a store's sorted rows.
#pragma once

#include "sp_graph.cuh"

namespace sp {

namespace {

// K searches in lockstep: pos[k] = entries of row old[k] (deg[k] entries,
// ascending cols in [0, n)) with a smaller col than col[k], present[k] = whether
// col[k] is there.  What a search costs is its dependent reads of random
// sectors, so each read takes the whole 32-byte sector (four entries: rows
// start on sector boundaries and hold a multiple of four slots), and the next
// sector is found by interpolation between the cols that bound what is left
// (the row's first and last to begin with, read together, so that it does not
// matter where in [0, n) a row's cols lie): three or four reads for evenly
// spread cols, however long the row, against one per halving.  After kGuesses
// of them every second read halves what is left, which bounds a search of
// unevenly spread cols by two reads per halving.
template <int K>
__device__ __forceinline__ void row_search(const int2 *const *old, const int *deg, const int *col,
                                           int n, u32 *pos, bool *present) {
  constexpr int kEnds = 4, kGuesses = 4;   // more sectors than kEnds: the row's ends first
  int lo[K], hi[K], xlo[K], xhi[K];   // sectors left, and the cols around them
#pragma unroll
  for (int k = 0; k < K; ++k) {
    lo[k] = 0;
    hi[k] = (deg[k] + 3) / 4;
    pos[k] = (u32)deg[k];
    present[k] = false;
    xlo[k] = hi[k] > kEnds ? __ldg(&old[k][0].x) : -1;
    xhi[k] = hi[k] > kEnds ? __ldg(&old[k][deg[k] - 1].x) : n;
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (hi[k] <= kEnds) continue;
    if (col[k] <= xlo[k]) {
      pos[k] = 0;
      present[k] = col[k] == xlo[k];
      hi[k] = 0;
    } else if (col[k] >= xhi[k]) {
      present[k] = col[k] == xhi[k];
      pos[k] = (u32)(deg[k] - (present[k] ? 1 : 0));
      hi[k] = 0;
    }
  }
  for (int it = 0;; ++it) {
    const bool guess = it < kGuesses || (it & 1);
    bool act = false;
    int g[K];
    int4 a[K], b[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int left = hi[k] - lo[k];
      act |= left > 0;
      int s = left >> 1;
      if (guess && left > 2) {
        s = (int)((float)(col[k] - xlo[k]) / (float)(xhi[k] - xlo[k]) * (float)left);
        s = max(0, min(s, left - 1));
      }
      g[k] = lo[k] + s;
      a[k] = b[k] = make_int4(0, 0, 0, 0);
      if (left > 0) {
        const int4 *p = (const int4 *)(old[k] + 4LL * g[k]);
        a[k] = __ldg(p);
        b[k] = __ldg(p + 1);
      }
    }
    if (!act) break;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int left = hi[k] - lo[k];
      if (left <= 0) continue;
      const int e = 4 * g[k], c = col[k];
      // (slots past the end of the row count as larger than every col)
      const int c0 = a[k].x;
      const int c1 = e + 1 < deg[k] ? a[k].z : n, c2 = e + 2 < deg[k] ? b[k].x : n;
      const int c3 = e + 3 < deg[k] ? b[k].z : n;
      if (c0 >= c) {           // the answer is here or before
        pos[k] = (u32)e;
        present[k] = c0 == c;
        hi[k] = c0 == c ? lo[k] : g[k];
        xhi[k] = c0;
      } else if (c3 < c) {
        lo[k] = g[k] + 1;
        xlo[k] = c3;
      } else {
        pos[k] = (u32)(e + 1 + (c1 < c) + (c2 < c));
        present[k] = c1 == c || c2 == c || c3 == c;
        hi[k] = lo[k];
      }
    }
  }
}

}  // namespace

}  // namespace sp
