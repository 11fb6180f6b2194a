// Elementwise passes of the backward sweep's lesser functions, one pair of transposed tiles per CTA.
//
// With PGL = P G^<_{i+1,i+1} and X2 = G_{i+1,i+1} Q the sweep needs
//     G^<_{i,i+1} = X2^H - PGL,   W = X2 - PGL^H / 2,   Re Tr[(H - E S)_{i,i+1} (G^<_{i,i+1})^H]
// and, with T = P W, G^<_ii = g^<_i + T - T^H, its trace and its complex128 copy.  A CTA takes tiles (I, J)
// and (J, I) of an energy, so every operand is read once (a pass of single tiles reads the transposed
// operand a second time) and both results, the traces and the output leave in the same pass: bound by HBM.
// The traces' partial sums are added in a fixed order by k_trace_sums.  At b = 256 and 96 energies in df32 the
// two passes replace 57 + 57 + 167 us of separate combinations and traces and half of the 63 us output pass.
#include <type_traits>

#include "df32.cuh"
#include "kernels.cuh"

namespace qtx {

namespace {

constexpr int TS = 32;  // tile edge; 256 threads = 32 columns x 8 rows

__device__ __forceinline__ df sub_t(df a, df b) { return df_sub(a, b); }
__device__ __forceinline__ float sub_t(float a, float b) { return a - b; }
__device__ __forceinline__ double sub_t(double a, double b) { return a - b; }
__device__ __forceinline__ df add_t(df a, df b) { return df_add(a, b); }
__device__ __forceinline__ float add_t(float a, float b) { return a + b; }
__device__ __forceinline__ double add_t(double a, double b) { return a + b; }
__device__ __forceinline__ df half_t(df a) { return mkdf(0.5f * a.hi, 0.5f * a.lo); }
__device__ __forceinline__ float half_t(float a) { return 0.5f * a; }
__device__ __forceinline__ double half_t(double a) { return 0.5 * a; }
// a - b^H, a + b with b^H: (re, -im)
template <typename T>
__device__ __forceinline__ cx<T> minus_conj(cx<T> a, cx<T> b) {
  cx<T> r;
  r.re = sub_t(a.re, b.re);
  r.im = add_t(a.im, b.im);
  return r;
}

// tile pair of a linear index over I <= J
__device__ __forceinline__ void pair_of(int q, int nt, int& I, int& J) {
  I = 0;
  while (q >= nt - I) {
    q -= nt - I;
    ++I;
  }
  J = I + q;
}

// Trace partials: df32 sums for df32 blocks without an overlap matrix (error-free FP32 steps: the FP64 pipe runs at
// 1/64 of the FP32 rate); with one, where H - E S is formed in FP64, and for the other types, FP64
template <typename T, bool OVERLAP>
struct PartialOf {
  using type = double;
};
template <>
struct PartialOf<df, false> {
  using type = df;
};
__device__ __forceinline__ void acc_add(double& a, double b) { a += b; }
__device__ __forceinline__ void acc_add(df& a, df b) { a = df_add(a, b); }
__device__ __forceinline__ double shfl_down(double v, int off) { return __shfl_down_sync(0xffffffffu, v, off); }
__device__ __forceinline__ df shfl_down(df v, int off) {
  return mkdf(__shfl_down_sync(0xffffffffu, v.hi, off), __shfl_down_sync(0xffffffffu, v.lo, off));
}
__device__ __forceinline__ void zero(double& a) { a = 0.0; }
__device__ __forceinline__ void zero(df& a) { a = mkdf(0.f, 0.f); }
// sum over the CTA's 256 threads, in thread 0
template <typename A>
__device__ __forceinline__ A cta_sum(A v) {
  __shared__ A red[8];
  for (int off = 16; off > 0; off >>= 1) acc_add(v, shfl_down(v, off));
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = v;
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < 8; ++w) acc_add(v, red[w]);
  return v;
}

template <typename T>
__device__ __forceinline__ void load_tile(cx<T> (*s)[TS + 1], const cx<T>* X, int b, int r0, int c0) {
  const int tx = threadIdx.x % TS, ty = threadIdx.x / TS;
#pragma unroll
  for (int q = 0; q < TS / 8; ++q) {
    const int r = r0 + ty + 8 * q, c = c0 + tx;
    if (r < b && c < b) s[ty + 8 * q][tx] = X[(long)r * b + c];
  }
}

// Re((H - E S) conj(u)) accumulated
__device__ __forceinline__ void trace_term(df& a, cx<double> h, cx<df> u) {
  a = df_add(a, df_add(df_mul(from_d<df>(h.re), u.re), df_mul(from_d<df>(h.im), u.im)));
}
template <typename T>
__device__ __forceinline__ void trace_term(double& a, cx<double> h, cx<T> u) {
  a += h.re * to_d(u.re) + h.im * to_d(u.im);
}

// OVERLAP: Sup is given
template <typename T, bool OVERLAP>
__global__ void __launch_bounds__(256) k_lesser_offdiag(const cx<T>* PGL, cx<T>* X2, cx<T>* GLu, const cx<double>* Hup,
                                                        const cx<double>* Sup, const double* E, int b, int nt,
                                                        typename PartialOf<T, OVERLAP>::type* part) {
  after_previous();
  using Acc = typename PartialOf<T, OVERLAP>::type;
  extern __shared__ __align__(16) unsigned char dsm[];
  cx<T>(*pij)[TS + 1] = reinterpret_cast<cx<T>(*)[TS + 1]>(dsm);
  cx<T>(*pji)[TS + 1] = pij + TS;
  cx<T>(*xij)[TS + 1] = pji + TS;
  cx<T>(*xji)[TS + 1] = xij + TS;
  const int e = blockIdx.y, tx = threadIdx.x % TS, ty = threadIdx.x / TS;
  const long o = (long)e * b * b;
  int I, J;
  pair_of(blockIdx.x, nt, I, J);
  load_tile<T>(pij, PGL + o, b, I * TS, J * TS);
  load_tile<T>(xij, X2 + o, b, I * TS, J * TS);
  if (I != J) {
    load_tile<T>(pji, PGL + o, b, J * TS, I * TS);
    load_tile<T>(xji, X2 + o, b, J * TS, I * TS);
  } else {
    pji = pij;
    xji = xij;
  }
  __syncthreads();
  Acc acc;
  zero(acc);
  const double Ee = OVERLAP ? E[e] : 0.0;
  for (int side = 0; side < (I == J ? 1 : 2); ++side) {
    const int r0 = (side ? J : I) * TS, c0 = (side ? I : J) * TS;
    cx<T>(*p)[TS + 1] = side ? pji : pij;
    cx<T>(*pt)[TS + 1] = side ? pij : pji;
    cx<T>(*x)[TS + 1] = side ? xji : xij;
    cx<T>(*xt)[TS + 1] = side ? xij : xji;
#pragma unroll
    for (int q = 0; q < TS / 8; ++q) {
      const int lr = ty + 8 * q, r = r0 + lr, c = c0 + tx;
      if (r >= b || c >= b) continue;
      const long at = (long)r * b + c;
      const cx<T> pv = p[lr][tx], xh = xt[tx][lr], ph = pt[tx][lr];
      cx<T> u;  // X2^H - PGL
      u.re = sub_t(xh.re, pv.re);
      u.im = sub_t(sub_t(T{}, xh.im), pv.im);
      if (GLu) GLu[o + at] = u;
      if (Hup) {
        cx<double> h = Hup[at];
        if (OVERLAP) h = h - Ee * Sup[at];
        trace_term(acc, h, u);
      }
      cx<T> hp;  // PGL^H / 2 before conjugation
      hp.re = half_t(ph.re);
      hp.im = half_t(ph.im);
      X2[o + at] = minus_conj(x[lr][tx], hp);
    }
  }
  if (Hup) {
    acc = cta_sum(acc);
    if (threadIdx.x == 0) part[(long)e * gridDim.x + blockIdx.x] = acc;
  }
}

// gl <- gl + T - T^H; out64 (complex128, batch stride so) a copy of it; part: the trace of its imaginary
// parts, one partial per diagonal tile (FP64)
template <typename T>
__global__ void __launch_bounds__(256) k_lesser_diag(cx<T>* gl, const cx<T>* X, cx<double>* out64, long so, int b, int nt,
                                                     double* part) {
  after_previous();
  extern __shared__ __align__(16) unsigned char dsm[];
  cx<T>(*tij)[TS + 1] = reinterpret_cast<cx<T>(*)[TS + 1]>(dsm);
  cx<T>(*tji)[TS + 1] = tij + TS;
  const int e = blockIdx.y, tx = threadIdx.x % TS, ty = threadIdx.x / TS;
  const long o = (long)e * b * b;
  int I, J;
  pair_of(blockIdx.x, nt, I, J);
  load_tile<T>(tij, X + o, b, I * TS, J * TS);
  if (I != J) load_tile<T>(tji, X + o, b, J * TS, I * TS);
  else tji = tij;
  __syncthreads();
  double tr = 0.0;
  for (int side = 0; side < (I == J ? 1 : 2); ++side) {
    const int r0 = (side ? J : I) * TS, c0 = (side ? I : J) * TS;
    cx<T>(*t)[TS + 1] = side ? tji : tij;
    cx<T>(*tt)[TS + 1] = side ? tij : tji;
#pragma unroll
    for (int q = 0; q < TS / 8; ++q) {
      const int lr = ty + 8 * q, r = r0 + lr, c = c0 + tx;
      if (r >= b || c >= b) continue;
      const long at = (long)r * b + c;
      cx<T> v = gl[o + at];
      v.re = add_t(v.re, t[lr][tx].re);
      v.im = add_t(v.im, t[lr][tx].im);
      v = minus_conj(v, tt[tx][lr]);
      gl[o + at] = v;
      if (out64) {
        cx<double> w;
        w.re = to_d(v.re);
        w.im = to_d(v.im);
        out64[(long)e * so + at] = w;
      }
      if (r == c) tr += to_d(v.im);
    }
  }
  if (I == J) {
    tr = cta_sum(tr);
    if (threadIdx.x == 0) part[(long)e * nt + I] = tr;
  }
}

// cur[e * ldcur] = -2 sum of energy e's partials (cur may be null), den[e * ldden] = sum of its others; one warp an
// energy, lanes take every 32nd partial and are added pairwise
template <typename Acc>
__global__ void k_trace_sums(double* cur, long ldcur, const Acc* pc, int nc, double* den, long ldden, const double* pd,
                             int nd) {
  after_previous();
  const int e = blockIdx.x, l = threadIdx.x;
  if (cur) {
    Acc a;
    zero(a);
    for (int i = l; i < nc; i += 32) acc_add(a, pc[(long)e * nc + i]);
    for (int off = 16; off > 0; off >>= 1) acc_add(a, shfl_down(a, off));
    if (l == 0) cur[(long)e * ldcur] = -2.0 * to_d(a);
  }
  double d = 0.0;
  for (int i = l; i < nd; i += 32) d += pd[(long)e * nd + i];
  for (int off = 16; off > 0; off >>= 1) d += shfl_down(d, off);
  if (l == 0) den[(long)e * ldden] = d;
}

inline int tiles_of(int b) { return (b + TS - 1) / TS; }

}  // namespace

size_t lesser_scratch_bytes(int b, int batch) {
  const size_t nt = tiles_of(b);
  return (size_t)batch * (nt * (nt + 1) / 2 + nt) * sizeof(double);
}

template <typename T, bool OVERLAP>
static cudaError_t launch_offdiag(const cx<T>* PGL, cx<T>* X2, cx<T>* GLu, const cx<double>* Hup, const cx<double>* Sup,
                                  const double* E, int b, int batch, void* scratch, cudaStream_t st) {
  const int nt = tiles_of(b);
  const int smem = 4 * TS * (TS + 1) * (int)sizeof(cx<T>);
  static std::atomic<unsigned long long> done{0};
  const cudaError_t e = allow_smem(k_lesser_offdiag<T, OVERLAP>, smem, done);
  if (e != cudaSuccess) return e;
  launch_after(k_lesser_offdiag<T, OVERLAP>, dim3(nt * (nt + 1) / 2, batch), 256, smem, st, PGL, X2, GLu, Hup, Sup, E, b, nt,
               reinterpret_cast<typename PartialOf<T, OVERLAP>::type*>(scratch));
  count_launch();
  return cudaGetLastError();
}
template <typename T>
cudaError_t lesser_offdiag(const cx<T>* PGL, cx<T>* X2, cx<T>* GLu, const cx<double>* Hup, const cx<double>* Sup,
                           const double* E, int b, int batch, void* scratch, cudaStream_t st) {
  return Hup && Sup ? launch_offdiag<T, true>(PGL, X2, GLu, Hup, Sup, E, b, batch, scratch, st)
                    : launch_offdiag<T, false>(PGL, X2, GLu, Hup, Sup, E, b, batch, scratch, st);
}

template <typename T>
cudaError_t lesser_diag(cx<T>* gl, const cx<T>* X, cx<double>* out64, long so, double* cur, long ldcur, bool overlap, double* den,
                        long ldden, int b, int batch, void* scratch, cudaStream_t st) {
  const int nt = tiles_of(b), np = nt * (nt + 1) / 2;
  double* pd = reinterpret_cast<double*>(scratch) + (size_t)batch * np;
  launch_after(k_lesser_diag<T>, dim3(np, batch), 256, 2 * TS * (TS + 1) * sizeof(cx<T>), st, gl, X, out64, so, b, nt, pd);
  count_launch();
  auto sums = [&](auto A) {
    using Acc = decltype(A);
    launch_after(k_trace_sums<Acc>, batch, 32, 0, st, cur, ldcur, reinterpret_cast<const Acc*>(scratch), np, den, ldden, pd, nt);
  };
  if (overlap) sums(typename PartialOf<T, true>::type{});
  else sums(typename PartialOf<T, false>::type{});
  count_launch();
  return cudaGetLastError();
}

#define QTX_LESSER(T)                                                                                                   \
  template cudaError_t lesser_offdiag<T>(const cx<T>*, cx<T>*, cx<T>*, const cx<double>*, const cx<double>*,           \
                                         const double*, int, int, void*, cudaStream_t);                                \
  template cudaError_t lesser_diag<T>(cx<T>*, const cx<T>*, cx<double>*, long, double*, long, bool, double*, long, int, int, \
                                      void*, cudaStream_t);
QTX_LESSER(double)
QTX_LESSER(float)
QTX_LESSER(df)
#undef QTX_LESSER

}  // namespace qtx
