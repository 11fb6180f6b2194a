// FP64 batched complex products on the tcgen05 tensor cores (sm_103a).
//
// C[e] = alpha * op(A[e]) * op(B[e]) + beta * C0[e]   (complex128 in and out)
//
// GB300's FP64 pipe gives 1.1 TFLOP/s, so a DFMA product of 256 x 256 blocks takes 130 us per batch
// entry.  Here every row of op(A) and column of op(B) is scaled by a power of two and rounded to a
// 62-bit integer (61 bits when K > 256), nine bits below the last place of the row's largest entry,
// and written as nine balanced base-128 digits in bf16 planes (Ozaki-style slicing, paper Sec. II-D).
// The 45 digit products with i + j <= 10 run as tcgen05.mma kind::f16 into eight TMEM accumulators:
//   acc0..acc6: i + j = 2..8, exact in FP32 (multiples of 2^(-7 (i+j-2)), below 2^24 units),
//   acc7:       i + j = 9, 10, below 2^-32 of the leading group: its FP32 rounding is below 2^-56.
// The epilogue converts the accumulators to integers, adds them in 92-bit fixed point and rounds to
// FP64 once, so a product carries one rounding of the whole sum plus the operands' 2^-62 (measured
// against 64-bit references: closer than the DFMA product, whose rounding errors grow with K).
//
// Why nine digits and eight accumulators: eight digits (36 products) drop digit products at 2^-51 of
// the result, as much as DFMA's own rounding; nine put the truncation near 2^-58.  Eight
// accumulators of 64 columns (32 complex columns, MMA N = 64, 24.8 ns each) fill the 512 TMEM
// columns; nine exact ones would leave 24 complex columns at nearly the same time per instruction.
//
// Rows or columns with an infinity or a NaN take digits of zero and are computed by the epilogue with
// DFMA from the operands themselves, so they propagate as in an FP64 product.
//
// Kernel structure: as the product kernel of tc_engine.cu (persistent, one CTA per SM, a producer
// warp of bulk copies, two MMA-issuing threads, eight epilogue warps, every wait bounded).
//
// What bounds it (products of 256^3): the MMAs, 46 cycles each with their operands read from shared
// memory (6 KB at 128 B per cycle: 48; the tensor core alone 32), 78% of an SM's time, and the
// recombination while it holds TMEM, 14%.
#include <cuda_bf16.h>

#include <atomic>
#include <type_traits>

#include "fix64.cuh"
#include "kernels.cuh"
#include "tc_ptx.cuh"

namespace qtx {
namespace tc {
namespace {

constexpr int S9 = kDig64;
constexpr int BNC9 = 32;                    // complex output columns per tile (MMA N = 64)
constexpr int NACC9 = 8;
constexpr int ACC9 = 2 * BNC9;              // TMEM columns of one accumulator
constexpr int SUB_B9 = BNC9 * BKS * 2;
constexpr int SLOT_A9 = S9 * TILE_A;       // the planes of a left tile's K-step (36 KB)
constexpr int SLOT_B9 = S9 * 3 * SUB_B9;   // the planes and parts of a right tile's K-block (27 KB)
constexpr int NSA9 = 3, NSB9 = 2;          // slots of the two rings
constexpr int RING9 = NSA9 * SLOT_A9 + NSB9 * SLOT_B9;
constexpr int OUT9 = BM * BNC9 * 16;        // staging: [BM][BNC9] complex128, XOR-swizzled
constexpr int SMEM9 = RING9 + OUT9 + (BM + BNC9) * 4 + 128;

struct Params {
  const unsigned char* pa;  // A [batch'][M_pad/128][K_pad/16][Re, Im][9][128 x 32 B]
  const unsigned char* pb;  // B [batch'][N_pad/32][K_pad/16][9][-Im, Re, Im][rows x 32 B], rows = 32 or bn_last
  const int *eA, *eB;
  int M_pad, N_pad, nks, M, N, K, bn_last, escale;
  int a_batched, b_batched;
  const cx<double>*A, *B;   // the operands (rows and columns with non-finite values)
  long lda, sA, ldb, sB;
  int opA, opB;
  cx<double>* C; long ldc, sC;
  const cx<double>* C0; long ldc0, sC0;
  double alpha, beta;
  int akind, bkind;         // alpha: 0 = +1, 1 = -1, 2 = general; beta the same, 3 = no C0 term
  const int* active;
  int NBt, MBt;
};
// A launch covers the tiles of 1..kMany9 products: product q owns tiles [tile0[q], tile0[q+1]), column tile
// fastest, then row tile, then batch entry.
constexpr int kMany9 = 4;
struct Launch {
  int n, hold;
  int* err;
  uint64_t limit_ns;
  int tile0[kMany9 + 1];
  Params p[kMany9];
};
// product of global tile t, and t's index within it
template <bool MANY>
__device__ __forceinline__ int product_of(const Launch& L, long t, int& lt) {
  int q = 0;
  if (MANY)
    while (q + 1 < L.n && t >= L.tile0[q + 1]) ++q;
  lt = (int)t - (MANY ? L.tile0[q] : 0);
  return q;
}

// the MMA thread that issues accumulator ga's digit products: 22 of the 45 one, 23 the other
__host__ __device__ constexpr int mma_half9(int ga) { return ga == 5 || ga == 7; }

__device__ __forceinline__ int at9(int r, int c) { return r * BNC9 + (c ^ (r & 7)); }

// one output value from the eight accumulators (pre-scaled digit products), times 2^Es
__device__ __forceinline__ double recombine(const uint32_t (&v)[NACC9][8], int c, int Es) {
  // exact groups as integers of their own unit 2^(-7 g); the tail in units of 2^-53
  auto fx = [&](int g, int sh) { return (int64_t)__float2int_rn(__uint_as_float(v[g][c]) * __int_as_float((127 + sh) << 23)); };
  const int64_t hi = (fx(0, 0) << 28) + (fx(1, 7) << 21) + (fx(2, 14) << 14) + (fx(3, 21) << 7) + fx(4, 28);
  const int64_t lo = (fx(5, 35) << 21) + (fx(6, 42) << 14) + (fx(7, 53) << 3);
  bool bad = false;
  const double x = fix_sum_scaled(hi, lo, Es, bad);
  return bad ? scale64(fix_sum(hi, lo), Es) : x;
}

// (op(A) op(B))(m, n) of one batch entry by DFMA: rows or columns with non-finite values
__device__ __noinline__ cx<double> dot_dfma(const Params& p, int e, int m, int n) {
  const cx<double>* A = p.A + (long)e * p.sA;
  const cx<double>* B = p.B + (long)e * p.sB;
  cx<double> acc = mk<double>(0.0, 0.0);
  for (int k = 0; k < p.K; ++k) {
    const cx<double> a = p.opA == OP_N ? A[(long)m * p.lda + k] : conj(A[(long)k * p.lda + m]);
    const cx<double> b = p.opB == OP_N ? B[(long)k * p.ldb + n] : conj(B[(long)n * p.ldb + k]);
    cfma(acc, a, b);
  }
  return acc;
}

template <bool MANY>
__global__ void __launch_bounds__(352, 1) k_tc_gemm_fp64(const __grid_constant__ Launch L) {
  const int n_tiles = L.tile0[L.n];
  extern __shared__ __align__(1024) unsigned char base[];
  unsigned char* ringB = base + NSA9 * SLOT_A9;
  cx<double>* out = reinterpret_cast<cx<double>*>(base + RING9);
  int* s_eA = reinterpret_cast<int*>(base + RING9 + OUT9);
  int* s_eB = s_eA + BM;
  uint64_t* fullA = reinterpret_cast<uint64_t*>(s_eB + BNC9);
  uint64_t* emptyA = fullA + NSA9;
  uint64_t* fullB = emptyA + NSA9;
  uint64_t* emptyB = fullB + NSB9;
  uint64_t* accf = emptyB + NSB9;
  uint64_t* acce = accf + 1;
  uint64_t* holdbar = acce + 1;   // never arrived at (the wait test)
  uint64_t* drainbar = acce + 2;  // the MMA thread's final commit
  uint32_t* tslot = reinterpret_cast<uint32_t*>(acce + 3);
  int* s_got = reinterpret_cast<int*>(tslot + 1);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NSA9; ++s) {
      mbar_init(&fullA[s], 1);
      mbar_init(&emptyA[s], 2);  // both MMA threads' commits
    }
    for (int s = 0; s < NSB9; ++s) {
      mbar_init(&fullB[s], 1);
      mbar_init(&emptyB[s], 2);
    }
    mbar_init(accf, 2);
    mbar_init(acce, 1);
    mbar_init(holdbar, 1);
    mbar_init(drainbar, 2);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // (the previous launch's CTAs may still hold TMEM, or wait for it: nothing is allocated before they end)
  after_previous();
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot;

  if (warp == 0) {
    if (lane == 0) {
      long ga = 0, gb = 0;  // copies into the left and the right ring so far
      bool ok = true;
      for (int k = 0; ok; ++k) {
        const long t = tile_at(k);
        if (t >= n_tiles) break;
        int lt;
        const Params& p = L.p[product_of<MANY>(L, t, lt)];
        const long MB = p.M_pad / BM, NB = p.N_pad / BNC9, nkb = p.nks / 2;
        const int e = lt / (p.NBt * p.MBt), mblk = (lt / p.NBt) % p.MBt, nblk = lt % p.NBt;
        if (p.active && !p.active[e]) continue;
        const long ea = p.a_batched ? e : 0, eb = p.b_batched ? e : 0;
        const uint32_t bytesB = S9 * 3u * (uint32_t)(nblk == p.NBt - 1 ? p.bn_last : BNC9) * BKS * 2;
        const unsigned char* srcA = p.pa + (ea * MB + mblk) * p.nks * (long)SLOT_A9;
        const unsigned char* srcB = p.pb + (eb * NB + nblk) * nkb * (long)SLOT_B9;
        for (int ks = 0; ks < p.nks; ++ks, ++ga) {
          if (!(ks & 1)) {
            const int s = (int)(gb % NSB9);
            if (!mbar_wait(&emptyB[s], ((uint32_t)(gb / NSB9) & 1u) ^ 1u, L.err, L.limit_ns)) { ok = false; break; }
            mbar_expect_tx(&fullB[s], bytesB);
            bulk_load(ringB + s * SLOT_B9, srcB + (ks / 2) * (long)bytesB, bytesB, &fullB[s]);
            ++gb;
          }
          const int s = (int)(ga % NSA9);
          if (!mbar_wait(&emptyA[s], ((uint32_t)(ga / NSA9) & 1u) ^ 1u, L.err, L.limit_ns)) { ok = false; break; }
          mbar_expect_tx(&fullA[s], SLOT_A9);
          bulk_load(base + s * SLOT_A9, srcA + ks * (long)SLOT_A9, SLOT_A9, &fullA[s]);
        }
      }
      // the last copies issued land before the CTA goes on to exit
      for (long g = ga > NSA9 ? ga - NSA9 : 0; g < ga; ++g)
        mbar_wait_drain(&fullA[g % NSA9], (uint32_t)(g / NSA9) & 1u, kWaitLimitNs);
      for (long g = gb > NSB9 ? gb - NSB9 : 0; g < gb; ++g)
        mbar_wait_drain(&fullB[g % NSB9], (uint32_t)(g / NSB9) & 1u, kWaitLimitNs);
    }
    __syncwarp();
  } else if (warp == 1 || warp == 10) {
    const int half = warp == 10;
    if (lane == 0) {
      long ga = 0, gb = 0;
      int j = 0;
      bool ok = true;
      if (L.hold && !mbar_wait(holdbar, 0u, L.err, L.limit_ns)) ok = false;
      for (int k = 0; ok; ++k) {
        const long t = tile_at(k);
        if (t >= n_tiles) break;
        int lt;
        const Params& p = L.p[product_of<MANY>(L, t, lt)];
        if (p.active && !p.active[lt / (p.NBt * p.MBt)]) continue;
        const uint32_t rows = lt % p.NBt == p.NBt - 1 ? p.bn_last : BNC9;
        const uint32_t idesc = idesc_n(2 * rows);
        const uint32_t part = rows * BKS * 2 / 16;  // a descriptor's address counts 16-byte units
        if (!mbar_wait(acce, ((uint32_t)j & 1u) ^ 1u, L.err, L.limit_ns)) break;
        fence_after();
        for (int ks = 0; ks < p.nks; ++ks, ++ga) {
          const int sb = (int)(gb % NSB9), sa = (int)(ga % NSA9);
          if (!(ks & 1) && !mbar_wait(&fullB[sb], (uint32_t)(gb / NSB9) & 1u, L.err, L.limit_ns)) { ok = false; break; }
          if (!mbar_wait(&fullA[sa], (uint32_t)(ga / NSA9) & 1u, L.err, L.limit_ns)) { ok = false; break; }
          fence_after();
          // A's real parts (even steps) meet the B rows (Re, Im), its imaginary parts (-Im, Re)
          const uint64_t ad = sdesc(su32(base + sa * SLOT_A9));
          const uint64_t bd = sdesc(su32(ringB + sb * SLOT_B9)) + ((ks & 1) ? 0 : part);
          auto issue = [&](auto H) {
#pragma unroll
            for (int i = 1; i <= S9; ++i) {
#pragma unroll
              for (int jj = 1; jj <= S9 + 1 - i; ++jj) {
                const int ga9 = i + jj - 2 < NACC9 - 1 ? i + jj - 2 : NACC9 - 1;
                if (mma_half9(ga9) != decltype(H)::value) continue;
                // the first product of an accumulator's first step overwrites it
                const bool first = i == 1 && jj == ga9 + 1;
                mma(tmem + ga9 * ACC9, ad + (i - 1) * TILE_A / 16, bd + (jj - 1) * 3 * part, idesc, first ? (uint32_t)(ks > 0) : 1u);
              }
            }
          };
          if (half) issue(std::integral_constant<int, 1>());
          else issue(std::integral_constant<int, 0>());
          mma_commit(&emptyA[sa]);
          if (ks & 1) {
            mma_commit(&emptyB[sb]);
            ++gb;
          }
        }
        if (!ok) break;
        mma_commit(accf);
        ++j;
      }
      mma_commit(drainbar);
      mbar_wait_drain(drainbar, 0u, kWaitLimitNs);
    }
    __syncwarp();
  } else {
    // epilogue: warps 2..9; TMEM lane quarter = warp % 4, alternate chunks of 8 columns by half
    const int q = warp & 3, h = (warp - 2) >> 2;
    const int r = q * 32 + lane;
    const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16);
    const int et = threadIdx.x - 64;
    int j = 0;
    for (int k = 0;; ++k) {
      const long t = tile_at(k);
      if (t >= n_tiles) break;
      int lt;
      const Params& p = L.p[product_of<MANY>(L, t, lt)];
      const int e = lt / (p.NBt * p.MBt), mblk = (lt / p.NBt) % p.MBt, nblk = lt % p.NBt;
      if (p.active && !p.active[e]) continue;
      const int bn = nblk == p.NBt - 1 ? p.bn_last : BNC9;
      __syncwarp();
      asm volatile("bar.sync 1, 256;" ::: "memory");  // the previous tile's staging area is free
      if (et < BNC9) s_eB[et] = p.eB[(long)(p.b_batched ? e : 0) * p.N_pad + nblk * BNC9 + et];
      if (et >= 64 && et < 64 + BM) s_eA[et - 64] = p.eA[(long)(p.a_batched ? e : 0) * p.M_pad + mblk * BM + et - 64];
      if (et == 0) *s_got = mbar_wait(accf, (uint32_t)j & 1u, L.err, L.limit_ns) ? 1 : 0;
      __syncwarp();
      asm volatile("bar.sync 2, 256;" ::: "memory");
      if (!*s_got) break;
      fence_after();
      const int er = s_eA[r] - p.escale;  // a non-finite row's or column's values are replaced below
#pragma unroll 1
      for (int c0 = 8 * h; c0 < bn; c0 += 16) {
#pragma unroll 1
        for (int part = 0; part < 2; ++part) {
          uint32_t v[NACC9][8];
#pragma unroll
          for (int g = 0; g < NACC9; ++g) tmem_ld8(trow + g * ACC9 + part * bn + c0, v[g]);
          tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < 8; ++c) (&out[at9(r, c0 + c)].re)[part] = recombine(v, c, er + s_eB[c0 + c]);
        }
      }
      fence_before();
      __syncwarp();
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (et == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(acce)) : "memory");
      // store phase, overlapping the next tile's MMAs: alpha, beta C0
      const cx<double>* C0e = p.C0 ? p.C0 + (long)e * p.sC0 : nullptr;
      cx<double>* Ce = p.C + (long)e * p.sC;
      for (int idx = et; idx < BM * bn; idx += 256) {
        const int rr = idx / bn, cc = idx % bn;
        const int m = mblk * BM + rr, n = nblk * BNC9 + cc;
        if (m >= p.M || n >= p.N) continue;
        cx<double> v = out[at9(rr, cc)];
        const int ea = s_eA[rr], eb = s_eB[cc];
        if (ea >= kExpoNonFinite || eb >= kExpoNonFinite) v = dot_dfma(p, e, m, n);
        if (p.akind == 1) v = mk<double>(-v.re, -v.im);
        else if (p.akind == 2) v = p.alpha * v;
        if (p.bkind != 3) {
          cx<double> c0 = C0e[(long)m * p.ldc0 + n];
          if (p.bkind == 1) c0 = mk<double>(-c0.re, -c0.im);
          else if (p.bkind == 2) c0 = p.beta * c0;
          v = v + c0;
        }
        Ce[(long)m * p.ldc + n] = v;
      }
      ++j;
    }
  }
  __syncwarp();
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

// ------------------------------------------------------------------------------ digit planes
// Row exponents and digit planes of one operand in one pass: a strip of RPC logical rows (rows of
// op(A), columns of op(B)) goes once from global to shared memory, one warp per row; each thread then
// turns 8 consecutive k of a row into nine 16-byte plane chunks per part.  Bound by HBM: it reads 16 B
// and writes 36 (left) or 54 B (right operand: Re, Im, -Im) per complex value.
__host__ __device__ constexpr int skew9(int k) { return k + (k >> 3); }

// Both operands of every product of a launch share one digitisation (blockIdx.z).
struct Operand {
  const cx<double>* X;
  long ldx, sX;
  int R, R_pad, K, K_pad, P, transposed, conj, batch;
  int* eout;
  unsigned char* planes;
  const int* active;
};
struct Operands {
  Operand o[2 * kMany9];  // left, right of each product
};
template <int RPC>
__global__ void __launch_bounds__(32 * RPC) k_digitize_fp64(const __grid_constant__ Operands ops) {
  after_previous();
  const int side = blockIdx.z & 1, e = blockIdx.y;
  const Operand& op = ops.o[blockIdx.z];
  const int K = op.K, K_pad = op.K_pad, P = op.P;
  const int R = op.R, R_pad = op.R_pad, transposed = op.transposed, conj_ = op.conj;
  const long ldx = op.ldx;
  if (e >= op.batch || (int)blockIdx.x * RPC >= R_pad || (op.active && !op.active[e])) return;
  extern __shared__ __align__(16) unsigned char dsm[];
  constexpr int NT = 32 * RPC;
  const int ldS = skew9(K_pad) + 1;
  cx<double>* strip = reinterpret_cast<cx<double>*>(dsm);
  __shared__ int s_ex[RPC];
  const cx<double>* Xe = op.X + (long)e * op.sX;
  int* eout = op.eout;
  const int r0 = blockIdx.x * RPC, t = threadIdx.x;
  if (t < RPC) s_ex[t] = kExpoZero;
  __syncthreads();
  const cx<double> zero = mk<double>(0.0, 0.0);
  // direct strips: threads along k (row by row); transposed ones: threads along the rows, then k
  const int rs = transposed ? t % RPC : 0, k1 = transposed ? t / RPC : t, kst = transposed ? NT / RPC : NT;
  for (int rr = rs; rr < RPC; rr += transposed ? RPC : 1) {
    const int r = r0 + rr;
    int mx = kExpoZero;
    for (int k0 = k1; k0 < K_pad; k0 += 4 * kst) {
      cx<double> v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int k = k0 + u * kst;
        v[u] = (r < R && k < K) ? Xe[transposed ? (long)k * ldx + r : (long)r * ldx + k] : zero;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int k = k0 + u * kst;
        if (k >= K_pad) break;
        strip[rr * ldS + skew9(k)] = v[u];
        mx = max(mx, max(expo64(v[u].re), expo64(v[u].im)));
      }
    }
    const int grp = transposed ? RPC : 1;  // lanes of a warp that hold the same row are grp apart
    for (int off = 16; off >= grp; off >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    if ((t & 31) < grp) atomicMax(&s_ex[rr], mx);
  }
  __syncthreads();
  if (t < RPC && r0 + t < R_pad) eout[(long)e * R_pad + r0 + t] = s_ex[t];
  // the layouts of Params::pa and Params::pb: each block is what one copy of the product kernel takes
  const int nkb = K_pad / BKS;
  unsigned char* pe = op.planes + (long)e * (side == 0 ? (long)(R_pad / BM) * 2 * nkb * SLOT_A9 : (long)(R_pad / BNC9) * nkb * SLOT_B9);
  const int nkc = K_pad / 8;
  const int R_wr = side == 1 ? min(R_pad, (R + 7) / 8 * 8) : R_pad;  // columns past bn_last are never read
#pragma unroll 1
  for (int item = t; item < RPC * nkc; item += NT) {
    const int rr = item / nkc, k8 = 8 * (item % nkc), r = r0 + rr;
    if (r >= R_wr) continue;
    const int ex = s_ex[rr];
    const bool dead = ex >= kExpoNonFinite;  // zero digits; the product kernel computes these by DFMA
    uint64_t vr[8], vi[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      cx<double> v = strip[rr * ldS + skew9(k8 + j)];
      if (conj_) v.im = -v.im;
      vr[j] = dead ? kDigBias : fix_biased(v.re, P - ex);
      vi[j] = dead ? kDigBias : fix_biased(v.im, P - ex);
    }
    unsigned char *pr, *pi, *pn = nullptr;  // the chunk of Re, Im and -Im in the first plane; bytes from plane to plane
    long step;
    if (side == 0) {
      pr = pe + ((long)(r / BM) * nkb + k8 / BKS) * 2 * SLOT_A9 + sw32_offset((uint32_t)(r % BM), (uint32_t)(k8 % BKS));
      pi = pr + SLOT_A9;
      step = TILE_A;
    } else {
      const int cb = r / BNC9, rows = cb == R_pad / BNC9 - 1 ? (R - cb * BNC9 + 7) / 8 * 8 : BNC9, part = rows * BKS * 2;
      pn = pe + (long)cb * nkb * SLOT_B9 + (long)(k8 / BKS) * (S9 * 3 * part) + sw32_offset((uint32_t)(r % BNC9), (uint32_t)(k8 % BKS));
      pr = pn + part;
      pi = pr + part;
      step = 3 * part;
    }
#pragma unroll
    for (int i = 0; i < S9; ++i) {
      const uint32_t sc = digit_scale(i), sh = digit_shift(i);
      auto word = [&](uint64_t a, uint64_t b) {
        const uint32_t w = 0x43004300u | digit_field(a, i) | (digit_field(b, i) << 16);
        const __nv_bfloat162 d = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&w), *reinterpret_cast<const __nv_bfloat162*>(&sc),
                                         *reinterpret_cast<const __nv_bfloat162*>(&sh));
        return *reinterpret_cast<const uint32_t*>(&d);
      };
      const uint4 re = make_uint4(word(vr[0], vr[1]), word(vr[2], vr[3]), word(vr[4], vr[5]), word(vr[6], vr[7]));
      const uint4 im = make_uint4(word(vi[0], vi[1]), word(vi[2], vi[3]), word(vi[4], vi[5]), word(vi[6], vi[7]));
      *reinterpret_cast<uint4*>(pr + i * step) = re;
      *reinterpret_cast<uint4*>(pi + i * step) = im;
      if (side == 1) {
        const uint32_t g = 0x80008000u;  // the bf16 sign bits
        *reinterpret_cast<uint4*>(pn + i * step) = make_uint4(im.x ^ g, im.y ^ g, im.z ^ g, im.w ^ g);
      }
    }
  }
}

// ------------------------------------------------------------------------------ host side
constexpr int kMaxK9 = 512;  // longest contraction of one launch (exactness of the leading groups)

struct Dims9 {
  int M_pad, N_pad, K_pad, l1, P;
  size_t a, b, ea, eb;  // bytes per batch entry
};
size_t al1k(size_t x) { return (x + 1023) & ~size_t(1023); }
Dims9 dims9(int M, int N, int K) {
  Dims9 d;
  d.M_pad = (M + BM - 1) / BM * BM;
  d.N_pad = (N + BNC9 - 1) / BNC9 * BNC9;
  d.K_pad = (K + 15) / 16 * 16;
  if (d.K_pad == 0) d.K_pad = 16;
  // the leading digit's magnitude (64, or 32 beyond 512 embedded K) keeps the groups through
  // i + j = 6 below 2^24 units whatever the data; later groups that exceed it (operands whose digits
  // all agree in sign) round at 2^-24 of a sum that is 2^-35 and less of such a product
  d.l1 = 2 * d.K_pad <= 512 ? 7 : 6;
  d.P = DW * (S9 - 1) + d.l1 - 1;
  d.a = al1k((size_t)S9 * d.M_pad * 2 * d.K_pad * 2);
  d.b = al1k((size_t)(d.N_pad / BNC9) * (d.K_pad / BKS) * SLOT_B9);
  d.ea = al1k((size_t)d.M_pad * sizeof(int));
  d.eb = al1k((size_t)d.N_pad * sizeof(int));
  return d;
}
int chunk_k(int K) {
  const int nc = (K + kMaxK9 - 1) / kMaxK9;
  return nc <= 1 ? K : (K + nc - 1) / nc;
}

// n products, each with `bytes` of scratch behind the last one's
cudaError_t products9(const GemmArgs<double>* g, int n, unsigned char* scratch, size_t bytes, int* err_flag, cudaStream_t st,
                      cudaEvent_t* ev) {
  cudaError_t e;
  Launch L;
  Operands o;
  L.n = n;
  L.hold = wait_test();
  L.limit_ns = L.hold ? kWaitTestLimitNs : kWaitLimitNs;
  L.err = err_flag;
  long tiles = 0;
  int R = 0, K_pad = 0, batch = 0;
  for (int q = 0; q < n; ++q) {
    const GemmArgs<double>& x = g[q];
    Params& p = L.p[q];
    const Dims9 d = dims9(x.M, x.N, x.K);
    const int ab = x.sA != 0, bb = x.sB != 0;
    const size_t na = ab ? x.batch : 1, nb = bb ? x.batch : 1;
    p.M_pad = d.M_pad;
    p.N_pad = d.N_pad;
    unsigned char* pa = scratch + (size_t)q * bytes;
    unsigned char* pb = pa + na * d.a;
    int* eA = reinterpret_cast<int*>(pb + nb * d.b);
    int* eB = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(eA) + na * d.ea);
    o.o[2 * q] = Operand{x.A, x.lda, x.sA, x.M, d.M_pad, x.K, d.K_pad, d.P, x.opA == OP_C, x.opA == OP_C, (int)na, eA, pa, ab ? x.active : nullptr};
    o.o[2 * q + 1] = Operand{x.B, x.ldb, x.sB, x.N, d.N_pad, x.K, d.K_pad, d.P, x.opB == OP_N, x.opB == OP_C, (int)nb, eB, pb, bb ? x.active : nullptr};
    R = R > d.M_pad ? R : d.M_pad;
    R = R > d.N_pad ? R : d.N_pad;
    K_pad = K_pad > d.K_pad ? K_pad : d.K_pad;
    batch = batch > x.batch ? batch : x.batch;
    p.pa = pa;
    p.pb = pb;
    p.eA = eA;
    p.eB = eB;
    p.nks = 2 * d.K_pad / BKS;
    p.M = x.M; p.N = x.N; p.K = x.K;
    p.escale = 2 * d.l1 - 2;
    p.a_batched = ab; p.b_batched = bb;
    p.A = x.A; p.B = x.B; p.lda = x.lda; p.sA = x.sA; p.ldb = x.ldb; p.sB = x.sB;
    p.opA = x.opA; p.opB = x.opB;
    p.C = x.C; p.ldc = x.ldc; p.sC = x.sC;
    p.C0 = x.C0; p.ldc0 = x.ldc0; p.sC0 = x.sC0;
    p.alpha = x.alpha; p.beta = x.beta;
    auto kind = [](double v) { return v == 1.0 ? 0 : (v == -1.0 ? 1 : 2); };
    p.akind = kind(x.alpha);
    p.bkind = (x.C0 && x.beta != 0.0) ? kind(x.beta) : 3;
    p.active = x.active;
    p.NBt = d.N_pad / BNC9;
    p.MBt = d.M_pad / BM;
    p.bn_last = (x.N - (p.NBt - 1) * BNC9 + 7) / 8 * 8;
    L.tile0[q] = (int)tiles;
    tiles += (long)p.NBt * p.MBt * x.batch;
    if (tiles > 0x7fffffffL) return cudaErrorInvalidValue;
  }
  L.tile0[n] = (int)tiles;
  constexpr int RPC = 4;  // transposed strips read four values of 16 bytes in a row: whole 32-byte sectors
  const size_t smem = (size_t)RPC * (skew9(K_pad) + 1) * sizeof(cx<double>);  // at most 37 KB
  launch_after(k_digitize_fp64<RPC>, dim3(R / RPC, batch, 2 * n), 32 * RPC, smem, st, o);
  count_launch();
  if ((e = cudaGetLastError())) return e;
  int sms = 0;
  static std::atomic<unsigned long long> done1{0}, done2{0};
  if ((e = n == 1 ? allow_smem(k_tc_gemm_fp64<false>, SMEM9, done1) : allow_smem(k_tc_gemm_fp64<true>, SMEM9, done2)) || (e = sm_count(sms))) return e;
  const unsigned grid = (unsigned)(tiles < sms ? tiles : sms);
  if (ev) cudaEventRecord(ev[0], st);
  if (n == 1) launch_after<1>(k_tc_gemm_fp64<false>, grid, 352, SMEM9, st, L);
  else launch_after<1>(k_tc_gemm_fp64<true>, grid, 352, SMEM9, st, L);
  count_launch();
  if (ev) cudaEventRecord(ev[1], st);
  return cudaGetLastError();
}

}  // namespace
}  // namespace tc

// scratch bytes of one batch entry (digit planes and exponents)
static size_t entry_bytes(int M, int N, int K) {
  const tc::Dims9 d = tc::dims9(M, N, tc::chunk_k(K));
  return d.a + d.b + d.ea + d.eb;
}

size_t gemm_fp64_tc_scratch_bytes(int M, int N, int K, int batch) {
  // enough entries for four waves of tiles, at most 384 MiB (but at least one entry): the batch is
  // taken in portions of what fits
  const size_t one = entry_bytes(M, N, K);
  const long tiles = (long)((M + tc::BM - 1) / tc::BM) * ((N + tc::BNC9 - 1) / tc::BNC9);
  size_t n = (size_t)((4 * kSms + tiles - 1) / tiles);
  const size_t cap = ((size_t)384 << 20) / one;
  if (n > cap) n = cap;
  if (n > (size_t)batch) n = (size_t)batch;
  return (n < 1 ? 1 : n) * one;
}

bool gemm_fp64_tc_fits(int M, int N, int K, size_t scratch_bytes) { return scratch_bytes >= entry_bytes(M, N, K); }

cudaError_t gemm_fp64_tc(const GemmArgs<double>& g0, void* scratch, size_t scratch_bytes, int* err_flag, cudaStream_t st,
                         cudaEvent_t* ev) {
  if (g0.M <= 0 || g0.N <= 0 || g0.batch <= 0) return cudaSuccess;
  const long room = (long)(scratch_bytes / entry_bytes(g0.M, g0.N, g0.K));
  if (room < 1 || g0.K < 1) return cudaErrorInvalidValue;
  const int Kc = tc::chunk_k(g0.K);
  // the events bracket the product kernel, or the whole call when it takes several launches
  const bool one = g0.batch <= room && g0.K <= Kc;
  if (ev && !one) cudaEventRecord(ev[0], st);
  for (long e0 = 0; e0 < g0.batch; e0 += room) {
    GemmArgs<double> g = g0;
    g.batch = (int)(g0.batch - e0 < room ? g0.batch - e0 : room);
    g.A += e0 * g.sA;
    g.B += e0 * g.sB;
    g.C += e0 * g.sC;
    if (g.C0) g.C0 += e0 * g.sC0;
    if (g.active) g.active += e0;
    // contractions beyond one launch's K run as consecutive chunks, each added to the last result
    for (int k0 = 0; k0 < g0.K; k0 += Kc) {
      GemmArgs<double> t = g;
      t.K = g0.K - k0 < Kc ? g0.K - k0 : Kc;
      t.A += g.opA == OP_N ? (long)k0 : (long)k0 * g.lda;
      t.B += g.opB == OP_N ? (long)k0 * g.ldb : (long)k0;
      if (k0 > 0) {
        t.C0 = g.C;
        t.ldc0 = g.ldc;
        t.sC0 = g.sC;
        t.beta = 1.0;
      }
      const cudaError_t e = tc::products9(&t, 1, reinterpret_cast<unsigned char*>(scratch), 0, err_flag, st, one ? ev : nullptr);
      if (e != cudaSuccess) return e;
    }
  }
  if (ev && !one) cudaEventRecord(ev[1], st);
  return cudaSuccess;
}

int gemm_fp64_tc_many(const GemmArgs<double>* g, int n, size_t scratch_bytes) {
  size_t most = 0;
  for (int q = 0; q < n; ++q) {
    if (g[q].M <= 0 || g[q].N <= 0 || g[q].K < 1 || g[q].batch <= 0 || tc::chunk_k(g[q].K) != g[q].K) return 1;
    const size_t need = entry_bytes(g[q].M, g[q].N, g[q].K) * g[q].batch;
    most = most > need ? most : need;
  }
  const size_t fit = most ? scratch_bytes / most : 1;
  const int k = fit < (size_t)tc::kMany9 ? (int)fit : tc::kMany9;
  return k < 1 ? 1 : (k < n ? k : n);
}

cudaError_t gemm_fp64_tc_launch(const GemmArgs<double>* g, int n, void* scratch, size_t scratch_bytes, int* err_flag, cudaStream_t st) {
  return tc::products9(g, n, reinterpret_cast<unsigned char*>(scratch), (scratch_bytes / n) & ~size_t(1023), err_flag, st, nullptr);
}

}  // namespace qtx
