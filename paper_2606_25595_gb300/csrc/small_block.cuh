// FP64 block arithmetic inside one CTA for blocks of at most 32 (the solve of small blocks, small.cu): products
// and inverses of complex128 blocks held in shared memory.
//
// GB300's FP64 pipe issues two DFMA a cycle and SM, so a product of two 16 x 16 complex blocks is
// 8,600 cycles of it.  Products here run on the tensor cores instead, as in tc_fp64.cu: each row of
// op(A) and column of op(B) becomes nine balanced base-128 digits in bf16 (62 bits of the row's
// largest entry), the 45 digit products with i + j <= 10 run as mma.sync m16n8k16 into eight exact (the
// last: i + j = 9, 10, rounded below 2^-56) FP32 accumulators, and the sum is rounded to FP64 once:
// about 1,700 cycles.  (mma.sync rather than tcgen05: a block is at most two 16-row tiles, a tcgen05
// tile has 128 rows, and the chain of dependent products of one energy leaves nothing to overlap a
// TMEM round trip with.)  Inverses start from FP32 Gauss-Jordan elimination and are refined with these
// products; a block beyond FP32's reach is eliminated in FP64.
//
// Layout: NM = 16 or 32 padded rows; an FP64 block is [NM][NM + 1] complex128 (the odd stride keeps
// row and column reads free of bank conflicts), zero outside the b x b block; digit planes are
// [9][NM rows or columns][2 NM + 8] bf16, k < NM real parts, NM <= k < 2 NM imaginary parts.
#pragma once
#include <cuda_bf16.h>

#include <type_traits>

#include "common.cuh"
#include "fix64.cuh"

namespace qtx {
namespace blk {

constexpr int kThreads = 256;
constexpr int kBufs = 8;  // FP64 blocks of the working set

template <int NM>
struct Smem {
  static constexpr int LD = NM + 1;
  static constexpr int PK = 2 * NM + 8;  // bf16 per plane row (16-byte rows, 8 rows in distinct bank groups)
  cx<double> m[kBufs][NM * LD];
  alignas(16) __nv_bfloat16 pa[kDig64][NM * PK];
  alignas(16) __nv_bfloat16 pb[kDig64][NM * PK];
  int ea[NM], eb[NM];
  int64_t xhi[4][2][32], xlo[8][2][32];  // NM = 16: halves of the sums, exchanged between warps w and w + 4
  int piv[NM], step[NM];
  unsigned norm;
  float fnorm[kThreads / 32];
  double red[kThreads / 32 * 2];
  // the FP32 elimination's two copies of the block share the left operand's planes
  __device__ cx<float>* f(int i) { return reinterpret_cast<cx<float>*>(pa) + i * NM * NM; }
  static_assert(2 * NM * NM * sizeof(cx<float>) <= sizeof(pa), "FP32 copies fit");
};

__device__ __forceinline__ uint32_t sm32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldsm2(uint32_t (&r)[2], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(a) : "memory");
}
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Digit planes of one operand: NM / 32 (or two per warp for NM = 16) logical rows at a time, one lane
// per k.  Row r is row r of op(X) (trans = 0: X[r][k], 1: X[k][r]), conjugated with cj.
template <int NM>
__device__ __forceinline__ void digitize(const cx<double>* X, int trans, int cj, __nv_bfloat16 (*pl)[NM * Smem<NM>::PK],
                                         int* ex) {
  constexpr int LD = Smem<NM>::LD, PK = Smem<NM>::PK;
  const int k = threadIdx.x % NM, odd = k & 1;
#pragma unroll
  for (int r = threadIdx.x / NM; r < NM; r += kThreads / NM) {
    cx<double> v = trans ? X[k * LD + r] : X[r * LD + k];
    if (cj) v.im = -v.im;
    const unsigned lanes = NM == 32 ? 0xffffffffu : 0xffffu << (threadIdx.x & 16);
    const int e = __reduce_max_sync(lanes, max(expo64(v.re), expo64(v.im)));
    if (k == 0) ex[r] = e;
    // even lanes take the real parts of (k, k + 1), odd lanes the imaginary parts of (k - 1, k)
    const double give = odd ? v.re : v.im;
    const double got = __shfl_xor_sync(0xffffffffu, give, 1);
    const double x0 = odd ? got : v.re, x1 = odd ? v.im : got;
    const bool dead = e >= kExpoNonFinite;  // zero digits; mm computes these by DFMA
    const uint64_t a = dead ? kDigBias : fix_biased(x0, kFix62 - e), b = dead ? kDigBias : fix_biased(x1, kFix62 - e);
    const int at = r * PK + (odd ? NM + k - 1 : k);
#pragma unroll
    for (int i = 0; i < kDig64; ++i) {
      const uint32_t w = 0x43004300u | digit_field(a, i) | (digit_field(b, i) << 16), sc = digit_scale(i), sh = digit_shift(i);
      *reinterpret_cast<__nv_bfloat162*>(&pl[i][at]) =
          __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&w), *reinterpret_cast<const __nv_bfloat162*>(&sc),
                  *reinterpret_cast<const __nv_bfloat162*>(&sh));
    }
  }
}

// Digit products of one warp: 16 x 8 real outputs, digit pairs with G0 <= i + j < G1 (i + j = 7 and 8 share
// the last accumulator) of one term a b over 16 k.  a, b: shared addresses of plane 0 for this lane.
template <int NM, int G0, int G1>
__device__ __forceinline__ void digit_mmas(float (&acc)[8][4], uint32_t a, uint32_t b, uint32_t neg) {
  constexpr uint32_t PL = NM * Smem<NM>::PK * 2;  // bytes of a plane
  constexpr int J1 = G1 < kDig64 ? G1 : kDig64;
  uint32_t bb[kDig64][2];
#pragma unroll
  for (int j = 0; j < J1; ++j) ldsm2(bb[j], b + j * PL);
#pragma unroll
  for (int i = 0; i < J1; ++i) {
    uint32_t aa[4];
    ldsm4(aa, a + i * PL);
#pragma unroll
    for (int v = 0; v < 4; ++v) aa[v] ^= neg;
#pragma unroll
    for (int j = 0; j < kDig64; ++j)
      if (i + j >= G0 && i + j < G1) mma16816(acc[i + j < 7 ? i + j : 7], aa, bb[j]);
  }
}
// Fixed-point parts of a sum, from groups 0..5 (units 2^-28 and 2^-56) and groups 6, 7 (units 2^-56): group
// g is a multiple of 2^(-7 g) below 2^22 units for K <= 32, read off as an integer by adding 1.5 2^23; the
// rounded tail is taken in units of 2^-48.
__device__ __forceinline__ int64_t unit_int(float acc, int sh) {
  return (int64_t)(__float_as_int(fmaf(acc, __int_as_float((127 + sh) << 23), 12582912.f)) - 0x4B400000);
}
__device__ __forceinline__ void parts_hi(const float (&acc)[8][4], int v, int64_t& hi, int64_t& lo) {
  hi = unit_int(acc[0][v], 0) * (1 << 28) + unit_int(acc[1][v], 7) * (1 << 21) + unit_int(acc[2][v], 14) * (1 << 14) +
       unit_int(acc[3][v], 21) * (1 << 7) + unit_int(acc[4][v], 28);
  lo = unit_int(acc[5][v], 35) * (1 << 21);
}
__device__ __forceinline__ int64_t parts_lo(const float (&acc)[8][4], int v) {
  return unit_int(acc[6][v], 42) * (1 << 14) + unit_int(acc[7][v], 48) * (1 << 8);
}

// The value of fixed-point parts hi, lo at (r, c) where the fast sum cannot form it: outside the normal range, or in a
// row or column that holds an infinity or a NaN, where one part of (op(A) op(B))(r, c) is formed by DFMA in ascending
// k from the operands themselves and propagates them as in the launched path's product.
template <int NM>
__device__ __noinline__ double rare_value(const Smem<NM>& s, const cx<double>* A, int opA, const cx<double>* B, int opB, int r, int c,
                                          int part, int b, int64_t hi, int64_t lo) {
  constexpr int LD = Smem<NM>::LD;
  const int ea = s.ea[r], eb = s.eb[c];
  if (ea < kExpoNonFinite && eb < kExpoNonFinite) return scale64(fix_sum(hi, lo), ea + eb - 12);
  cx<double> acc = mk<double>(0.0, 0.0);
  if (r < b && c < b)
    for (int k = 0; k < b; ++k)
      cfma(acc, opA == OP_N ? A[r * LD + k] : conj(A[k * LD + r]), opB == OP_N ? B[k * LD + c] : conj(B[c * LD + k]));
  return part ? acc.im : acc.re;
}

// C = sign op(A) op(B) (+ C0) (+ diag I on the first b rows), all blocks in shared memory.  C may be C0, and A or
// B where both are finite.  da / db: digitise A / B (false: its planes are those of the last product with it on
// that side).
// Begins on operands that every thread has written before a barrier; ends with one.  Not inlined: the
// kernels call it from some twenty places, and inlined copies miss the instruction cache on every call.
//
// NM = 32: a warp owns one 16 x 8 complex tile.  NM = 16: four warps would own one part of a 16 x 8 tile
// each; warps w and w + 4 share it, one taking the digit groups 0-5, the other 6 and 7 (42 and 48 of the
// 90 products), and each rounds two of a lane's four values.
template <int NM>
__device__ __noinline__ void mm(Smem<NM>& s, int b, cx<double>* C, double sign, const cx<double>* A, int opA, const cx<double>* B, int opB,
                   const cx<double>* C0, double diag, bool da, bool db) {
  constexpr int LD = Smem<NM>::LD, PK = Smem<NM>::PK;
  if (da) digitize<NM>(A, opA == OP_C, opA == OP_C, s.pa, s.ea);
  if (db) digitize<NM>(B, opB == OP_N, opB == OP_C, s.pb, s.eb);
  __syncthreads();
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int mt = NM == 32 ? warp / 4 : 0, nt = NM == 32 ? warp % 4 : warp % 2;
  const uint32_t arow = sm32(&s.pa[0][(mt * 16 + lane % 16) * PK + (lane / 16) * 8]);
  const uint32_t brow = sm32(&s.pb[0][(nt * 8 + lane % 8) * PK + ((lane / 8) % 2) * 8]);
  constexpr uint32_t SGN = 0x80008000u;  // the bf16 sign bits
  // N of the lane's values v0, v0 + 1, ..: rounded together (the sums are free of branches), then stored
  auto put = [&](auto N, int v0, int part, const int64_t* hi, const int64_t* lo) {
    constexpr int n = decltype(N)::value;
    double x[n];
    bool bad = false;
#pragma unroll
    for (int q = 0; q < n; ++q) {
      const int v = v0 + q, r = mt * 16 + lane / 4 + (v / 2) * 8, c = nt * 8 + (lane % 4) * 2 + (v & 1);
      const int ex = s.ea[r] + s.eb[c];
      x[q] = fix_sum_scaled(hi[q], lo[q], ex - 12, bad);
      bad |= ex >= kExpoNonFinite / 2;
    }
#pragma unroll
    for (int q = 0; q < n; ++q) {
      const int v = v0 + q, r = mt * 16 + lane / 4 + (v / 2) * 8, c = nt * 8 + (lane % 4) * 2 + (v & 1);
      if (bad) x[q] = rare_value<NM>(s, A, opA, B, opB, r, c, part, b, hi[q], lo[q]);
      if (sign < 0) x[q] = -x[q];
      if (C0) x[q] += (&C0[r * LD + c].re)[part];
      if (diag != 0.0 && part == 0 && r == c && r < b) x[q] += diag;
      (&C[r * LD + c].re)[part] = x[q];
    }
  };
  float acc[8][4];
  auto clear = [&]() {
#pragma unroll
    for (int g = 0; g < 8; ++g)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[g][v] = 0.f;
  };
  if constexpr (NM == 32) {
#pragma unroll 1
    for (int part = 0; part < 2; ++part) {  // re: Ar Br - Ai Bi; im: Ar Bi + Ai Br
      clear();
#pragma unroll 1
      for (int k0 = 0; k0 < (b > 16 ? 32 : 16); k0 += 16) {
        digit_mmas<NM, 0, 9>(acc, arow + k0 * 2, brow + (part * NM + k0) * 2, 0u);
        digit_mmas<NM, 0, 9>(acc, arow + (NM + k0) * 2, brow + ((part ^ 1) * NM + k0) * 2, part ? 0u : SGN);
      }
      int64_t hi[4], lo[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        parts_hi(acc, v, hi[v], lo[v]);
        lo[v] += parts_lo(acc, v);
      }
      put(std::integral_constant<int, 4>(), 0, part, hi, lo);
    }
  } else {
    const int part = (warp / 2) % 2, t = warp % 4;
    clear();
    if (warp < 4) {
      digit_mmas<NM, 0, 6>(acc, arow, brow + part * NM * 2, 0u);
      digit_mmas<NM, 0, 6>(acc, arow + NM * 2, brow + (part ^ 1) * NM * 2, part ? 0u : SGN);
      int64_t hi[4], lo[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) parts_hi(acc, v, hi[v], lo[v]);
#pragma unroll
      for (int v = 2; v < 4; ++v) {
        s.xhi[t][v - 2][lane] = hi[v];
        s.xlo[t][v - 2][lane] = lo[v];
      }
      asm volatile("bar.sync %0, 64;" ::"r"(1 + t) : "memory");
#pragma unroll
      for (int v = 0; v < 2; ++v) lo[v] += s.xlo[4 + t][v][lane];
      put(std::integral_constant<int, 2>(), 0, part, hi, lo);
    } else {
      digit_mmas<NM, 6, 9>(acc, arow, brow + part * NM * 2, 0u);
      digit_mmas<NM, 6, 9>(acc, arow + NM * 2, brow + (part ^ 1) * NM * 2, part ? 0u : SGN);
      int64_t lo[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) lo[v] = parts_lo(acc, v);
#pragma unroll
      for (int v = 0; v < 2; ++v) s.xlo[4 + t][v][lane] = lo[v];
      asm volatile("bar.sync %0, 64;" ::"r"(1 + t) : "memory");
      int64_t hi[2];
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        hi[v] = s.xhi[t][v][lane];
        lo[2 + v] += s.xlo[t][v][lane];
      }
      put(std::integral_constant<int, 2>(), 2, part, hi, lo + 2);
    }
  }
  __syncthreads();
}

template <int NM>
__device__ __forceinline__ void load_block(cx<double>* D, const cx<double>* G, int b) {
  constexpr int LD = Smem<NM>::LD;
  for (int i = threadIdx.x; i < NM * NM; i += kThreads) {
    const int r = i / NM, c = i % NM;
    D[r * LD + c] = (r < b && c < b) ? G[r * b + c] : mk<double>(0.0, 0.0);
  }
}
template <int NM>
__device__ __forceinline__ void store_block(cx<double>* G, const cx<double>* D, int b) {
  constexpr int LD = Smem<NM>::LD;
  for (int i = threadIdx.x; i < NM * NM; i += kThreads) {
    const int r = i / NM, c = i % NM;
    if (r < b && c < b) G[r * b + c] = D[r * LD + c];
  }
}
// f(r, c, element index) over the b x b block
template <int NM, typename F>
__device__ __forceinline__ void each(int b, F f) {
  for (int i = threadIdx.x; i < NM * NM; i += kThreads) {
    const int r = i / NM, c = i % NM;
    if (r < b && c < b) f(r, c);
  }
}

// Frobenius norm of a block in FP32 (values beyond its range give infinity; all threads get it)
template <int NM>
__device__ __noinline__ float norm32(Smem<NM>& s, const cx<double>* X) {
  constexpr int LD = Smem<NM>::LD;
  float t = 0.f;
  for (int i = threadIdx.x; i < NM * NM; i += kThreads) {
    const cx<double> x = X[(i / NM) * LD + i % NM];
    const float a = __double2float_rn(x.re), c = __double2float_rn(x.im);
    t = fmaf(a, a, fmaf(c, c, t));
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
  if (threadIdx.x % 32 == 0) s.fnorm[threadIdx.x / 32] = t;
  __syncthreads();
  t = 0.f;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) t += s.fnorm[w];
  __syncthreads();
  return sqrtf(t);
}

// 1 / a in FP32 by |a|^2 of the value scaled to a magnitude in [1, 3) (a starting value: a few units)
__device__ __forceinline__ cx<float> recip32(cx<float> a) {
  const unsigned m = __float_as_uint(fmaxf(fabsf(a.re), fabsf(a.im))) & 0x7f800000u;
  const float sc = __uint_as_float(0x7f000000u - (m < 0x7f000000u ? m : 0x7e800000u));  // 2^-exponent
  const float x = a.re * sc, y = a.im * sc;
  const float r = __fdividef(sc, fmaf(x, x, y * y));
  return mk<float>(x * r, -y * r);
}

// FP32 Gauss-Jordan inverse of A (n x n) into X, one element (NM = 16) or four (NM = 32) per thread, the
// block in shared memory twice so that a step needs one barrier.  Pivot: the first largest |re| + |im| of
// the unused rows, found by every warp for itself.  Returns false (uniformly) for a zero or non-finite one.
template <int NM>
__device__ __noinline__ bool inverse_f32(Smem<NM>& s, cx<double>* X, const cx<double>* A, int n) {
  constexpr int LD = Smem<NM>::LD, PER = NM * NM / kThreads;
  const int c = threadIdx.x % NM, r0 = threadIdx.x / NM, lane = threadIdx.x % 32;
  cx<float> a[PER];
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int r = r0 + q * (kThreads / NM);
    const cx<double> v = A[r * LD + c];
    a[q] = mk<float>((float)v.re, (float)v.im);
    s.f(0)[r * NM + c] = a[q];
  }
  __syncthreads();
  unsigned used = 0;
  for (int k = 0; k < n; ++k) {
    const cx<float>* M = s.f(k & 1);
    unsigned key = 0;
    if (lane < n && !((used >> lane) & 1u)) {
      const cx<float> v = M[lane * NM + k];
      key = __float_as_uint(fabsf(v.re) + fabsf(v.im));
    }
    const unsigned best = __reduce_max_sync(0xffffffffu, key);
    if (best == 0 || best >= 0x7f800000u) return false;
    const int p = __ffs((int)__ballot_sync(0xffffffffu, key == best)) - 1;
    used |= 1u << p;
    if (threadIdx.x == 0) {
      s.piv[k] = p;
      s.step[p] = k;
    }
    const cx<float> w = recip32(M[p * NM + k]);
    const cx<float> pc = c == k ? w : M[p * NM + c] * w;
    cx<float>* N = s.f((k & 1) ^ 1);
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int r = r0 + q * (kThreads / NM);
      if (r == p) {
        a[q] = pc;
      } else {
        const cx<float> f = M[r * NM + k];
        cx<float> v = c == k ? mk<float>(0.f, 0.f) : a[q];
        v.re = fmaf(-f.re, pc.re, v.re);
        v.re = fmaf(f.im, pc.im, v.re);
        v.im = fmaf(-f.re, pc.im, v.im);
        v.im = fmaf(-f.im, pc.re, v.im);
        a[q] = v;
      }
      N[r * NM + c] = a[q];
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int r = r0 + q * (kThreads / NM);
    if (r < n && c < n) X[s.step[r] * LD + s.piv[c]] = mk<double>((double)a[q].re, (double)a[q].im);
    else X[r * LD + c] = mk<double>(0.0, 0.0);
  }
  __syncthreads();
  return true;
}

// FP64 Gauss-Jordan with partial pivoting in place (the blocks that refinement cannot resolve).
template <int NM>
__device__ __noinline__ bool eliminate(Smem<NM>& s, cx<double>* A, int n) {
  constexpr int LD = Smem<NM>::LD;
  const int t = threadIdx.x;
  for (int k = 0; k < n; ++k) {
    if (t < 32) {
      double best = (t >= k && t < n) ? cabs1(A[t * LD + k]) : -1.0;
      int at = t;
      for (int off = 16; off > 0; off >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, best, off);
        const int oi = __shfl_xor_sync(0xffffffffu, at, off);
        if (ov > best || ov != ov || (ov == best && oi < at)) {
          best = ov;
          at = oi;
        }
      }
      if (t == 0) s.piv[k] = (best > 0.0 && isfinite(best)) ? at : -1;
    }
    __syncthreads();
    const int p = s.piv[k];
    if (p < 0) return false;
    const cx<double> w = crecip(A[p * LD + k]);
    __syncthreads();
    if (t < n) {
      const cx<double> x = A[p * LD + t], y = A[k * LD + t];
      A[p * LD + t] = y;
      A[k * LD + t] = t == k ? w : x * w;
    }
    __syncthreads();
    cx<double> v[NM * NM / kThreads];
#pragma unroll
    for (int q = 0; q < NM * NM / kThreads; ++q) {
      const int i = t / NM + q * (kThreads / NM), j = t % NM;
      const cx<double> x = j == k ? mk<double>(0.0, 0.0) : A[i * LD + j];
      v[q] = i == k ? A[k * LD + j] : x - A[i * LD + k] * A[k * LD + j];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NM * NM / kThreads; ++q) {
      const int i = t / NM + q * (kThreads / NM), j = t % NM;
      if (i < n && j < n) A[i * LD + j] = v[q];
    }
    __syncthreads();
  }
  for (int k = n - 1; k >= 0; --k) {
    const int p = s.piv[k];
    if (p != k && t < n) {
      const cx<double> x = A[t * LD + k];
      A[t * LD + k] = A[t * LD + p];
      A[t * LD + p] = x;
    }
    __syncthreads();
  }
  return true;
}

// X = A^-1 (n x n blocks; R, T scratch; all four distinct; replaces every digit plane).  FP32 start, then Newton sweeps: with
// R = I - A X, one last X + X R from ||R|| <= 2^-27 on, X + (X + X R) R from 6e-6 on (the residual becomes
// its square or cube, 2e-16 at most); blocks that six sweeps do not bring
// there are eliminated in FP64.  Returns false for a zero or non-finite pivot.
template <int NM>
__device__ __noinline__ bool inverse(Smem<NM>& s, cx<double>* X, const cx<double>* A, cx<double>* R, cx<double>* T, int n) {
  constexpr int LD = Smem<NM>::LD;
  if (inverse_f32<NM>(s, X, A, n)) {
    for (int it = 0; it < 6; ++it) {
      mm<NM>(s, n, R, -1.0, A, OP_N, X, OP_N, nullptr, 1.0, true, true);
      const float nrm = norm32<NM>(s, R);
      if (nrm <= 0x1p-27f) {
        mm<NM>(s, n, X, 1.0, X, OP_N, R, OP_N, X, 0.0, true, true);
        return true;
      }
      if (nrm <= 6e-6f) {
        mm<NM>(s, n, T, 1.0, X, OP_N, R, OP_N, X, 0.0, true, true);
        mm<NM>(s, n, X, 1.0, T, OP_N, R, OP_N, X, 0.0, true, false);
        return true;
      }
      if (!(nrm < 0.9f)) break;
      mm<NM>(s, n, X, 1.0, X, OP_N, R, OP_N, X, 0.0, true, true);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < NM * NM; i += kThreads) X[(i / NM) * LD + i % NM] = A[(i / NM) * LD + i % NM];
  __syncthreads();
  return eliminate<NM>(s, X, n);
}

// sums of two per-thread values over the CTA (valid in thread 0; barriers inside).  Lanes 0-15 of a warp
// fold a, lanes 16-31 b: five FP64 additions a warp for both (each holds the FP64 pipe for 64 cycles).
template <int NM>
__device__ __noinline__ void sum2(Smem<NM>& s, double& a, double& b) {
  const int lane = threadIdx.x % 32, up = lane / 16;
  double x = (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
#pragma unroll
  for (int off = 8; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  __syncthreads();
  if (lane % 16 == 0) s.red[up * (kThreads / 32) + threadIdx.x / 32] = x;
  __syncthreads();
  if (threadIdx.x < 32) {
    x = s.red[lane % 16];
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    a = __shfl_sync(0xffffffffu, x, 0);
    b = __shfl_sync(0xffffffffu, x, 8);
  }
}

}  // namespace blk
}  // namespace qtx
