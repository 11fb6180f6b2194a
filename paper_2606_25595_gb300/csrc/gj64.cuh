// Pivot search and reciprocal of the FP64 Gauss-Jordan eliminations (leaf64.cu, decim.cu).  GB300's FP64
// pipe takes 64 cycles for a warp's instruction whatever its lanes do (measured), so one warp searches
// with integer compares and forms the reciprocal for its CTA, in two divisions (520 cycles each).
#pragma once
#include "common.cuh"

namespace qtx {
namespace gj {

// idx / n for idx < n^2, n <= 64 (exact: idx n < 2^20)
struct FastDiv {
  int n;
  unsigned m;
  __host__ __device__ explicit FastDiv(int n_) : n(n_), m((1u << 20) / (unsigned)n_ + 1u) {}
  __host__ __device__ int div(int idx) const { return (int)((unsigned)idx * m >> 20); }
};

// |re| + |im| as an integer that orders like it (NaN below everything)
__device__ __forceinline__ unsigned long long pivot_key(cx<double> a) {
  const unsigned long long v = (unsigned long long)__double_as_longlong(cabs1(a));
  return v <= 0x7ff0000000000000ull ? v : 0ull;
}
// largest key over the warp's lanes
__device__ __forceinline__ unsigned long long warp_max(unsigned long long key) {
  const unsigned h = __reduce_max_sync(0xffffffffu, (unsigned)(key >> 32));
  const unsigned l = __reduce_max_sync(0xffffffffu, (unsigned)(key >> 32) == h ? (unsigned)key : 0u);
  return ((unsigned long long)h << 32) | l;
}

// 1 / a by Smith's scaling (the operations of crecip, in their order), the last two divisions as one in
// two lanes.  Called by a whole warp with the same a.
__device__ __forceinline__ cx<double> crecip_warp(cx<double> a) {
  const int lane = threadIdx.x & 31;
  const bool tall = ((unsigned long long)__double_as_longlong(a.re) << 1) >= ((unsigned long long)__double_as_longlong(a.im) << 1);
  const double p = tall ? a.im : a.re, q = tall ? a.re : a.im;
  const double r = p / q, d = __fma_rn(p, r, q);
  const double num = tall ? (lane ? -r : 1.0) : (lane ? -1.0 : r);
  const double x = num / d;
  return mk<double>(__shfl_sync(0xffffffffu, x, 0), __shfl_sync(0xffffffffu, x, 1));
}

}  // namespace gj
}  // namespace qtx
