// Pivot search and reciprocal of the FP64 Gauss-Jordan eliminations (leaf64.cu, decim.cu).  GB300's FP64
// pipe takes 64 cycles for a warp's instruction whatever its lanes do (measured), so one warp searches
// with integer compares and forms the reciprocal for its CTA, in two divisions (520 cycles each).
#pragma once
#include "df32.cuh"

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

// Quotient a / b from y = 1 / b (1 + e), |e| < 2^-43 (a remainder correction, Markstein, IBM J. Res. Dev. 34, 111
// (1990)): q + rem y is within e^2 < 2^-86 of the quotient before its one rounding, so the result is the rounded
// quotient unless that lies as close to the middle of two FP64 numbers (as 1/b does for b one ulp below a power
// of two), where it may be the other of the two.
__device__ __forceinline__ double div_by(double a, double b, double y) {
  const double q = __dmul_rn(a, y);
  return __fma_rn(__fma_rn(-b, q, a), y, q);
}
// 1 / v to about 2^-45: the rounded reciprocal of v.hi and two terms of its error's series
__device__ __forceinline__ df recip_df(df v) {
  const float x = __frcp_rn(v.hi);
  const float e = __fmaf_rn(-v.lo, x, __fmaf_rn(-v.hi, x, 1.f));
  const float c = __fmul_rn(x, __fmaf_rn(e, e, e)), hi = __fadd_rn(x, c);
  return mkdf(hi, __fsub_rn(c, __fsub_rn(hi, x)));
}
// hi + lo of a normal df32 value, times +-2^s, without the FP64 pipe's conversions
__device__ __forceinline__ double widen(df v, int s, unsigned sign) {
  auto d = [&](float x) {
    const unsigned u = __float_as_uint(x);
    const int ex = (int)((u >> 23) & 255u);
    return ex ? __hiloint2double((int)((((u & 0x80000000u) ^ sign)) | ((unsigned)(ex + 896 + s) << 20) | ((u >> 3) & 0xfffffu)), (int)(u << 29)) : 0.0;
  };
  return __dadd_rn(d(v.hi), d(v.lo));
}

// 1 / a by Smith's scaling (the operations of crecip, in their order), the last two divisions as one in
// two lanes.  Called by a whole warp with the same a.
//
// A chain of FP64 instructions of 64 cycles each, in the way of every elimination step.  The two divisions
// (520 cycles each) take their reciprocals, 1/q and 1/d = q / (p^2 + q^2), from FP32 pairs, formed side by side
// before the first (the decimation of 4 energies at b = 16: 944 -> 883 us).  Operands outside the range where
// every step stays normal take the plain divisions.
__device__ __forceinline__ cx<double> crecip_warp(cx<double> a) {
  const int lane = threadIdx.x & 31;
  const unsigned long long M = 0x7fffffffffffffffull;
  const unsigned long long ur = (unsigned long long)__double_as_longlong(a.re) & M, ui = (unsigned long long)__double_as_longlong(a.im) & M;
  const bool tall = ur >= ui;
  const double p = tall ? a.im : a.re, q = tall ? a.re : a.im;
  const unsigned long long up = tall ? ui : ur, uq = tall ? ur : ui;
  const int ep = (int)(up >> 52), eq = (int)(uq >> 52);
  double x;
  if (eq > 223 && eq < 1823 && ep + 60 > eq) {
    // |p| and |q| over 2^(eq - 1023) as FP32 pairs
    auto pair = [](unsigned long long u, int s) {
      const unsigned long long m = (u & 0xfffffffffffffull) | 0x10000000000000ull;
      return mkdf(__fmul_rn((float)(unsigned)(m >> 29), __int_as_float((127 - 23 + s) << 23)),
                  __fmul_rn((float)(unsigned)(m & 0x1fffffffull), __int_as_float((127 - 52 + s) << 23)));
    };
    const df P = pair(up, ep - eq), Q = pair(uq, 0);
    const unsigned sign = (unsigned)(__double_as_longlong(q) >> 32) & 0x80000000u;
    const double y = widen(recip_df(Q), 1023 - eq, sign);
    const double w = widen(df_mul(Q, recip_df(df_add(df_mul(P, P), df_mul(Q, Q)))), 1023 - eq, sign);
    const double r = div_by(p, q, y), d = __fma_rn(p, r, q);
    x = div_by(tall ? (lane ? -r : 1.0) : (lane ? -1.0 : r), d, w);
  } else {
    const double r = p / q, d = __fma_rn(p, r, q);
    x = (tall ? (lane ? -r : 1.0) : (lane ? -1.0 : r)) / d;
  }
  return mk<double>(__shfl_sync(0xffffffffu, x, 0), __shfl_sync(0xffffffffu, x, 1));
}

}  // namespace gj
}  // namespace qtx
