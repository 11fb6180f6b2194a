// FP64 inverse of blocks of at most 64: Gauss-Jordan elimination with partial pivoting (the pivot is the
// first unused row of largest |Re| + |Im| in the column; rows stay where they are and the result is
// scattered at the end, as in k_leaf_inverse), one CTA per block, the block twice in shared memory.
//
// Bound by GB300's FP64 pipe (two DFMA a cycle and SM): 4 n^2 DFMA a step, 4,600 cycles at n = 48, after a
// chain of about 1,700 cycles for the pivot, its reciprocal and the scaled row.  Holding the rows in the
// registers of fixed warps and letting every warp form its own candidate's reciprocal took 640 us for a
// 48 x 48 block: eight reciprocals a step share the pipe, and lanes beyond n work on zeros.  Here one warp
// forms them, and the threads share the n^2 entries evenly (in registers, with a copy in shared memory for
// the pivot search and the factors).  The order of every rounding is that of the
// FP32 kernel's source and is written out.
#include "gj64.cuh"
#include "kernels.cuh"

namespace qtx {

namespace {

constexpr int kT = 512;

// LARGE: blocks above 32, whose pivot row's imaginary parts round the other product first
template <bool LARGE>
__global__ void __launch_bounds__(kT) k_leaf_fp64(cx<double>* Ag, long lda, long sA, const gj::FastDiv fd, const int* active,
                                                  int* status) {
  constexpr int NMAX = LARGE ? 64 : 32, PER = NMAX * NMAX / kT;
  const int e = blockIdx.x;
  if (active && !active[e]) return;
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ cx<double> rowk[NMAX];
  __shared__ int s_step[NMAX], s_piv[NMAX], s_p;
  const int n = fd.n, LD = n | 1, t = threadIdx.x;
  cx<double>* A = reinterpret_cast<cx<double>*>(dsm);
  cx<double>* B = A + n * LD;
  cx<double>* G = Ag + (long)e * sA;
  cx<double> x[PER];  // this thread's entries idx = t + kT m
#pragma unroll
  for (int m = 0; m < PER; ++m) {
    const int idx = t + kT * m, i = fd.div(idx), j = idx - i * n;
    if (idx < n * n) A[i * LD + j] = x[m] = G[(long)i * lda + j];
  }
  __syncthreads();
  unsigned long long used = 0;
  for (int k = 0; k < n; ++k) {
    if (t < 32) {
      const unsigned long long k0 = (t < n && !((used >> t) & 1)) ? gj::pivot_key(A[t * LD + k]) : 0ull;
      unsigned long long k1 = 0;
      if (LARGE) k1 = (t + 32 < n && !((used >> (t + 32)) & 1)) ? gj::pivot_key(A[(t + 32) * LD + k]) : 0ull;
      const unsigned long long best = gj::warp_max(k0 > k1 ? k0 : k1);
      const unsigned b0 = __ballot_sync(0xffffffffu, k0 == best), b1 = __ballot_sync(0xffffffffu, k1 == best);
      const bool ok = best != 0 && best < 0x7ff0000000000000ull;
      const int p = ok ? (b0 ? __ffs((int)b0) - 1 : 31 + __ffs((int)b1)) : -1;
      if (t == 0) s_p = p;
      if (ok) {
        const cx<double> r = gj::crecip_warp(A[p * LD + k]);
#pragma unroll
        for (int j = t; j < NMAX; j += 32) {
          if (j >= n) break;
          const cx<double> y = A[p * LD + j];
          const double im = LARGE ? __fma_rn(y.re, r.im, __dmul_rn(y.im, r.re)) : __fma_rn(y.im, r.re, __dmul_rn(y.re, r.im));
          rowk[j] = j == k ? r : mk<double>(__fma_rn(y.re, r.re, -__dmul_rn(y.im, r.im)), im);
        }
        if (t == 0) {
          s_step[p] = k;
          s_piv[k] = p;
        }
      }
    }
    __syncthreads();
    const int p = s_p;
    if (p < 0) {
      if (t == 0 && status) atomicCAS(status + e, 0, (int)QTX_ERR_SINGULAR);
      return;
    }
    used |= 1ull << p;
    // the pivot column -(f r), by the last warps
    cx<double> col = mk<double>(0.0, 0.0);
    const int ci = t - (kT - NMAX);
    if (ci >= 0 && ci < n) {
      const cx<double> f = A[ci * LD + k], r = rowk[k];
      col = mk<double>(-__fma_rn(f.re, r.re, -__dmul_rn(f.im, r.im)), -__fma_rn(f.re, r.im, __dmul_rn(f.im, r.re)));
    }
#pragma unroll
    for (int m = 0; m < PER; ++m) {
      const int idx = t + kT * m;
      if (idx - t >= n * n) break;  // uniform: whole rounds only
      if (idx < n * n) {
        const int i = fd.div(idx), j = idx - i * n;
        const cx<double> f = A[i * LD + k], a = rowk[j];
        cx<double> v = x[m];
        v.re = __fma_rn(-f.re, a.re, v.re);
        v.re = __fma_rn(f.im, a.im, v.re);
        v.im = __fma_rn(-f.re, a.im, v.im);
        v.im = __fma_rn(-f.im, a.re, v.im);
        x[m] = i == p ? a : v;
        if (j != k) B[i * LD + j] = x[m];
      }
    }
    if (ci >= 0 && ci < n) B[ci * LD + k] = ci == p ? rowk[k] : col;
    __syncthreads();
    // the column's owners take it back
#pragma unroll
    for (int m = 0; m < PER; ++m) {
      const int idx = t + kT * m;
      if (idx - t >= n * n) break;
      if (idx < n * n && idx - fd.div(idx) * n == k) x[m] = B[fd.div(idx) * LD + k];
    }
    cx<double>* q = A;
    A = B;
    B = q;
  }
#pragma unroll
  for (int m = 0; m < PER; ++m) {
    const int idx = t + kT * m, i = fd.div(idx), j = idx - i * n;
    if (idx < n * n) G[(long)s_step[i] * lda + s_piv[j]] = x[m];
  }
}

template <bool LARGE>
cudaError_t launch(cx<double>* A, long lda, long sA, int n, int batch, const int* active, int* status, cudaStream_t st) {
  constexpr int kMaxSmem = 2 * kLeafMax * (kLeafMax + 1) * (int)sizeof(cx<double>);
  static std::atomic<unsigned long long> done{0};
  const cudaError_t e = allow_smem(k_leaf_fp64<LARGE>, kMaxSmem, done);
  if (e != cudaSuccess) return e;
  k_leaf_fp64<LARGE><<<batch, kT, 2 * (size_t)n * (n | 1) * sizeof(cx<double>), st>>>(A, lda, sA, gj::FastDiv(n), active, status);
  count_launch();
  return cudaGetLastError();
}

}  // namespace

template <>
cudaError_t leaf_inverse<double>(cx<double>* A, long lda, long sA, int n, int batch, const int* active, int* status,
                                 cudaStream_t st) {
  if (n <= 0 || n > kLeafMax) return cudaErrorInvalidValue;
  return n <= 32 ? launch<false>(A, lda, sA, n, batch, active, status, st)
                 : launch<true>(A, lda, sA, n, batch, active, status, st);
}

}  // namespace qtx
