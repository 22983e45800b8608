// sp_acc.cuh -- a sum of |a - b| over 32-bit floats, at least as exact as one
// kept in 64 bits.  Plain C++ but for the rounding intrinsics, so that the host
// can compile it too.
//
// The GPU adds 64-bit floats at 1/64 of the rate of 32-bit ones, so the sum is
// kept as hi + mid + lo with error-free additions (Knuth's TwoSum: s = a + b
// rounded, e = its error, s + e = a + b exactly).  Nothing is rounded but lo, which
// holds the errors of mid, which holds the errors of hi: about 72 bits where the
// 64-bit sum has 53.  (With hi and lo only, 48 bits.)
#pragma once

#ifdef __CUDACC__
#define SP_ACC_FN __host__ __device__ __forceinline__
#else
#define SP_ACC_FN inline
#endif

namespace sp {

namespace {

struct Acc {
  float hi = 0.0f, mid = 0.0f, lo = 0.0f;
};

SP_ACC_FN float acc_plus(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}

// a + b, and the rounding error of that in *e.
SP_ACC_FN float two_sum(float a, float b, float *e) {
  const float s = acc_plus(a, b), z = acc_plus(s, -a);
  *e = acc_plus(acc_plus(a, -acc_plus(s, -z)), acc_plus(b, -z));
  return s;
}

SP_ACC_FN void acc_diff(Acc &c, float a, float b) {
  float e, x, y, z;
  const float d = two_sum(a, -b, &e);   // a - b = d + e exactly, e much the smaller
  c.hi = two_sum(c.hi, d < 0.0f ? -d : d, &x);
  c.mid = two_sum(c.mid, x, &y);
  c.mid = two_sum(c.mid, d < 0.0f ? -e : e, &z);
  c.lo = acc_plus(c.lo, acc_plus(y, z));
}

SP_ACC_FN void acc_merge(Acc &c, const Acc &o) {
  float x, y, z;
  c.hi = two_sum(c.hi, o.hi, &x);
  c.mid = two_sum(c.mid, o.mid, &y);
  c.mid = two_sum(c.mid, x, &z);
  c.lo = acc_plus(acc_plus(c.lo, o.lo), acc_plus(y, z));
}

SP_ACC_FN double acc_value(const Acc &c) {
  return (double)c.hi + ((double)c.mid + (double)c.lo);
}

}  // namespace

}  // namespace sp
