// Fixed-point helpers of the FP64 products on the tensor cores: an FP64 value as nine balanced
// base-128 digits, and the exact 92-bit sum of the digit products back as an FP64 value.  Integer
// operations only (GB300's FP64 pipe runs at 1/64 of the FP32 rate).
#pragma once
#include <stdint.h>
#include <string.h>

namespace qtx {

constexpr int kDig64 = 9;          // digits per FP64 operand value
constexpr int kFix62 = 62;         // P of nine digits with a leading one of at most 64
constexpr int kExpoNonFinite = 1 << 20;  // row exponent of a row that holds an infinity or a NaN
constexpr int kExpoZero = -4000;         // row exponent of a row of zeros

// sum_i 64 128^i: added to v, the 7-bit fields of the sum are the balanced digits plus 64
constexpr uint64_t kDigBias = 0x4081020408102040ull;

__host__ __device__ inline uint64_t bits_of(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t u;
  memcpy(&u, &x, 8);
  return u;
#endif
}
__host__ __device__ inline double double_of(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double x;
  memcpy(&x, &u, 8);
  return x;
#endif
}

// Exponent e with |x| < 2^e (subnormals: that of the smallest normal); kExpoZero for 0,
// kExpoNonFinite for infinities and NaN.
__host__ __device__ inline int expo64(double x) {
  const uint64_t u = bits_of(x) & 0x7fffffffffffffffull;
  const int ex = (int)(u >> 52);
  if (ex == 0x7ff) return kExpoNonFinite;
  if (u == 0) return kExpoZero;
  return (ex ? ex : 1) - 1022;
}

// round(x 2^(P - e)) (|x| < 2^e, P <= 62) plus the digit bias; ties away from zero.
__host__ __device__ inline uint64_t fix_biased(double x, int P_minus_e) {
  const uint64_t u = bits_of(x);
  if ((u << 1) == 0) return kDigBias;
  int ex = (int)((u >> 52) & 0x7ff);
  uint64_t m = u & ((1ull << 52) - 1);
  if (ex) m |= 1ull << 52;
  else ex = 1;
  const int sh = ex - 1075 + P_minus_e;  // at most P - 53
  uint64_t v;
  if (sh >= 0) v = m << sh;
  else if (sh > -54) v = (m + (1ull << (-sh - 1))) >> -sh;
  else v = 0;
  return ((u >> 63) ? 0 - v : v) + kDigBias;
}
// digit i (0 = leading) of a biased fixed-point value, plus 64: in [0, 127], the leading one in [0, 128]
__host__ __device__ inline uint32_t digit_field(uint64_t biased, int i) {
  return (uint32_t)(biased >> (7 * (kDig64 - 1 - i))) & (i == 0 ? 255u : 127u);
}

// bf16 pairs of 2^(-7 i) and -192 2^(-7 i): 0x4300 | (d + 64) is the bf16 of 192 + d (also for d = 64, where
// the OR carries into the exponent: 256), and (192 + d) s - 192 s = d s is exact in one bf16 FMA
__host__ __device__ constexpr uint32_t digit_scale(int i) { return (uint32_t)(127 - 7 * i) << 7 | (uint32_t)(127 - 7 * i) << 23; }
__host__ __device__ constexpr uint32_t digit_shift(int i) {
  return 0x80408040u | (uint32_t)(134 - 7 * i) << 7 | (uint32_t)(134 - 7 * i) << 23;
}

// RN((A 2^28 + B) 2^(Es - 56)) for |A| < 2^62, |B| < 2^62: the sum aligned to a 64-bit significand with a
// sticky bit, rounded to 53 bits, ties to even.  Free of branches, so that several sums interleave; `bad`
// is raised when the result is not a normal number (the caller then takes fix_sum and scale64).
__host__ __device__ inline double fix_sum_scaled(int64_t A, int64_t B, int Es, bool& bad) {
  const int64_t h0 = A + (B >> 28);
  const uint32_t l0 = (uint32_t)B << 4;  // 28 fraction bits at the top of a word
  const int64_t s = h0 >> 63;            // all ones if negative: (h0, l0) negated in two's complement
  const uint32_t l1 = (l0 ^ (uint32_t)s) - (uint32_t)s;
  const uint64_t h1 = (uint64_t)(h0 ^ s) - (uint64_t)(l0 == 0 ? s : 0);
  const bool small = h1 == 0;
  const uint64_t h = small ? (uint64_t)l1 << 32 : h1;
  const uint64_t l = small ? 0 : (uint64_t)l1 << 32;
  const bool zero = h == 0;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)(h | 1));
#else
  const int lz = __builtin_clzll((unsigned long long)(h | 1));
#endif
  const uint64_t m = (h << lz) | ((l >> 1) >> (63 - lz));
  const uint64_t r = m >> 11;
  const uint32_t odd = ((l << lz) != 0) | ((uint32_t)r & 1u);
  const uint32_t up = ((uint32_t)m & 0x7ffu) + odd > 0x400u;
  // exponent of the leading bit in units of 2^-28: 63 - lz, or -1 - lz when the word came from l1
  const int E = (small ? -1 : 63) - lz - 28 + 1022 + Es;
  bad |= !zero && (E < 0 || E > 2044);
  // r in [2^52, 2^53]: adding it to the exponent field minus one carries into the exponent
  const uint64_t u = ((uint64_t)(int64_t)E << 52) + r + up;
  return double_of(zero ? 0 : (u | ((uint64_t)s & 0x8000000000000000ull)));
}
// RN((A 2^28 + B) 2^-56)
__host__ __device__ inline double fix_sum(int64_t A, int64_t B) {
  bool bad = false;
  return fix_sum_scaled(A, B, 0, bad);
}

// x 2^E by its exponent field; results outside the normal range by two exact-or-rounding-once steps
#ifdef __CUDA_ARCH__
static __device__ __noinline__ double scale_rare(double x, int E) { return scalbn(x, E); }
__device__ __forceinline__ double scale64(double x, int E) {
  const uint64_t u = bits_of(x);
  const int ex = (int)((u >> 52) & 0x7ff) + E;
  if ((u << 1) == 0) return x;
  if (ex < 1 || ex > 2046) return scale_rare(x, E);
  return double_of(u + ((uint64_t)(int64_t)E << 52));
}
#else
__device__ double scale64(double x, int E);
#endif

}  // namespace qtx
