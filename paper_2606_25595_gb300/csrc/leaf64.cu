// FP64 inverse of blocks of at most 64: Gauss-Jordan elimination with partial pivoting (the pivot is the
// first unused row of largest |Re| + |Im| in the column; rows stay where they are and the result is
// scattered at the end, as in k_leaf_inverse), one cluster of 1, 2, 4 or 8 CTAs per block, each with a range of
// its columns in shared memory.
//
// Bound by GB300's FP64 pipe: a warp's instruction takes its quarter of the SM 64 cycles, whatever its lanes
// do.  4 n^2 DFMA a step are 4,600 cycles of one SM at n = 48, beside a chain of about 2,200 for the next
// column's update, its pivot, the reciprocal (two divisions of 520) and their way to the other CTAs.  So the
// columns are split over as many SMs as the batch leaves idle, and the chain runs ahead: in the CTA that owns
// column k + 1, warp 0 takes step k for that column alone, finds the pivot and the reciprocal and writes them
// with the column into every CTA, while the other warps make step k of their columns in place, 32 entries of one
// formula at a time (column k apart); in clusters of 4 and 8 they leave warp 0 its quarter of the SM, as the
// chain then decides.  One cluster barrier a step.  24 blocks of 48: 199 us in one CTA each, 104 us in clusters
// of 4.
// The order of every rounding is that of the FP32 kernel's source and is written out.
#include <cooperative_groups.h>

#include "gj64.cuh"
#include "kernels.cuh"

namespace qtx {

namespace {

namespace cg = cooperative_groups;
constexpr int kT = 256;

// What a step needs of its column: the entries before it, the pivot's row (-1: none) and reciprocal.
struct LeafStep {
  cx<double> f[kLeafMax], r;
  int p;
};

// LARGE: blocks above 32, whose pivot row's imaginary parts round the other product first
template <bool LARGE>
__global__ void __launch_bounds__(kT) k_leaf_fp64(cx<double>* Ag, long lda, long sA, int n, const int* active, int* status) {
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank(), e = blockIdx.x / C, t = threadIdx.x;
  if (active && !active[e]) return;
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ LeafStep s_col[2];
  __shared__ cx<double> rowk[kLeafMax];
  __shared__ int s_step[kLeafMax], s_piv[kLeafMax];
  const int c0 = rank * n / C, nc = (rank + 1) * n / C - c0;  // this CTA's columns
  const gj::FastDiv fd0(nc), fd1(nc > 1 ? nc - 1 : 1), fd2(nc > 2 ? nc - 2 : 1);
  // the warps of the update; warp 4 shares a quarter of the SM, and so its FP64 pipe, with warp 0
  const bool shared_pipe = C <= 2;
  const int w = t / 32, slots = shared_pipe ? 7 : 6, slot = shared_pipe || w < 4 ? w - 1 : (w == 4 ? -1 : w - 2);
  cx<double>* A = reinterpret_cast<cx<double>*>(dsm);  // [n][nc]
  cx<double>* G = Ag + (long)e * sA;
  auto sync = [&]() {
    if (C > 1) cl.sync();
    else __syncthreads();
  };
  for (int idx = t; idx < n * nc; idx += kT) A[idx] = G[(long)fd0.div(idx) * lda + c0 + idx - fd0.div(idx) * nc];
  auto scaled = [](cx<double> y, cx<double> r) {
    const double im = LARGE ? __fma_rn(y.re, r.im, __dmul_rn(y.im, r.re)) : __fma_rn(y.im, r.re, __dmul_rn(y.re, r.im));
    return mk<double>(__fma_rn(y.re, r.re, -__dmul_rn(y.im, r.im)), im);
  };
  auto update = [](cx<double> v, cx<double> f, cx<double> a) {
    v.re = __fma_rn(-f.re, a.re, v.re);
    v.re = __fma_rn(f.im, a.im, v.re);
    v.im = __fma_rn(-f.re, a.im, v.im);
    v.im = __fma_rn(-f.im, a.re, v.im);
    return v;
  };
  unsigned long long used = 0;
  // warp 0 of column k's owner: the column after step k - 1 (st; nullptr before the first), its pivot and
  // reciprocal, to every CTA of the cluster
  auto lead = [&](int k, const LeafStep* st) {
    const int j = k - c0;
    cx<double> v[2] = {mk<double>(0.0, 0.0), mk<double>(0.0, 0.0)};
    cx<double> a = mk<double>(0.0, 0.0);
    if (st) a = scaled(A[st->p * nc + j], st->r);
    unsigned long long key[2] = {0, 0};
    __syncwarp();
#pragma unroll
    for (int h = 0; h < (LARGE ? 2 : 1); ++h) {
      const int i = t + 32 * h;
      if (i >= n) break;
      v[h] = A[i * nc + j];
      if (st) A[i * nc + j] = v[h] = i == st->p ? a : update(v[h], st->f[i], a);
      if (!((used >> i) & 1)) key[h] = gj::pivot_key(v[h]);
    }
    __syncwarp();
    const unsigned long long best = gj::warp_max(key[0] > key[1] ? key[0] : key[1]);
    const unsigned b0 = __ballot_sync(0xffffffffu, key[0] == best), b1 = __ballot_sync(0xffffffffu, key[1] == best);
    const bool ok = best != 0 && best < 0x7ff0000000000000ull;
    const int p = ok ? (b0 ? __ffs((int)b0) - 1 : 31 + __ffs((int)b1)) : -1;
    cx<double> r = mk<double>(0.0, 0.0);
    if (ok) {
      const cx<double> x = p < 32 ? v[0] : v[1];
      r = gj::crecip_warp(mk<double>(__shfl_sync(0xffffffffu, x.re, p & 31), __shfl_sync(0xffffffffu, x.im, p & 31)));
    }
    for (int q = 0; q < C; ++q) {
      LeafStep* d = C > 1 ? cl.map_shared_rank(&s_col[k & 1], q) : &s_col[k & 1];
      if (t < n) d->f[t] = v[0];
      if (LARGE && t + 32 < n) d->f[t + 32] = v[1];
      if (t == 0) {
        d->p = p;
        d->r = r;
      }
    }
  };
  sync();  // every CTA has its columns (from here on others' shared memory and G are written)
  if (t < 32 && rank == 0) lead(0, nullptr);
  sync();
  for (int k = 0; k < n; ++k) {
    const LeafStep& st = s_col[k & 1];
    const int p = st.p;
    if (p < 0) {  // in every CTA alike
      if (t == 0 && rank == 0 && status) atomicCAS(status + e, 0, (int)QTX_ERR_SINGULAR);
      return;
    }
    used |= 1ull << p;
    const int k1 = k + 1 < n ? k + 1 - c0 : -1, kc = k - c0;  // columns k + 1 and k here, if within [0, nc)
    if (t < 32) {
      if (t == 0) {
        s_step[p] = k;
        s_piv[k] = p;
      }
      if (k1 >= 0 && k1 < nc) lead(k + 1, &st);
    } else if (slot >= 0) {
      const int u = t - 32;
      if (u < nc && u != k1) rowk[u] = u == kc ? st.r : scaled(A[p * nc + u], st.r);
      if (shared_pipe) asm volatile("bar.sync 1, 224;" ::: "memory");
      else asm volatile("bar.sync 1, 192;" ::: "memory");
      // 32 entries at a time of the columns but k and k + 1, then of column k
      const bool own0 = kc >= 0 && kc < nc, own1 = k1 >= 0 && k1 < nc;
      const int lo = own0 ? kc : k1;  // the columns left out here: lo, and lo + 1 if both are
      const gj::FastDiv& fx = own0 && own1 ? fd2 : (own0 || own1 ? fd1 : fd0);
      const int nx = nc - own0 - own1, items = nx > 0 ? (n * nx + 31) / 32 : 0, all = items + (own0 ? (n + 31) / 32 : 0);
      const int lane = t & 31;
      for (int it = slot; it < all; it += slots) {
        if (it < items) {
          const int idx = 32 * it + lane, i = fx.div(idx);
          int j = idx - i * nx;
          if (i >= n) continue;
          if ((own0 || own1) && j >= lo) j += own0 + own1;
          const cx<double> a = rowk[j], v = update(A[i * nc + j], st.f[i], a);
          A[i * nc + j] = i == p ? a : v;
        } else {
          const int i = 32 * (it - items) + lane;
          if (i >= n) continue;
          const cx<double> f = st.f[i], r = st.r;
          const cx<double> v = mk<double>(-__fma_rn(f.re, r.re, -__dmul_rn(f.im, r.im)), -__fma_rn(f.re, r.im, __dmul_rn(f.im, r.re)));
          A[i * nc + kc] = i == p ? r : v;
        }
      }
    }
    sync();
  }
  for (int idx = t; idx < n * nc; idx += kT) {
    const int i = fd0.div(idx), j = idx - i * nc;
    G[(long)s_step[i] * lda + s_piv[c0 + j]] = A[idx];
  }
}

template <bool LARGE>
cudaError_t launch(cx<double>* A, long lda, long sA, int n, int batch, const int* active, int* status, cudaStream_t st) {
  static std::atomic<unsigned long long> done{0};
  const cudaError_t e = allow_smem(k_leaf_fp64<LARGE>, kLeafMax * kLeafMax * (int)sizeof(cx<double>), done);
  if (e != cudaSuccess) return e;
  // CTAs of a cluster: as many as leave every block resident at once on the SMs, with columns for each
  int C = 1;
  while (C < 8 && (long)batch * C * 2 <= kSms && 8 * C < n) C *= 2;
  const size_t smem = (size_t)n * ((n + C - 1) / C) * sizeof(cx<double>);
  EarlyLaunches none(0);  // (clusters that wait on SMs early: contacts of b = 48 in 12.0 instead of 9.5 ms)
  const cudaError_t le = launch_after_clusters(k_leaf_fp64<LARGE>, C, batch * C, kT, smem, st, A, lda, sA, n, active, status);
  count_launch();
  return le != cudaSuccess ? le : cudaGetLastError();
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
