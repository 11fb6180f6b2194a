// Contact self-energies by Sancho-Rubio decimation (Lopez Sancho et al., J. Phys. F 15, 851 (1985)),
// FP64, without host synchronisation.
//
// For a lead with principal layer H00 and coupling H01 (from a lead cell to the next one away from
// the device), per energy z = E + i eta:
//     alpha = H01, beta = H01^H, eps = eps_s = H00;
//     repeat:  g = (z - eps)^-1
//              eps_s += alpha g beta,  eps += alpha g beta + beta g alpha,
//              alpha = alpha g alpha,  beta = beta g beta
//     until max |alpha|, |beta| < tol max |H01|;  then g_s = (z - eps_s)^-1 and
//     Sigma^R = H01 g_s H01^H  (the device's end slice couples to the first lead cell by H01).
//
// k_decimate: the whole iteration of one energy and contact in one cluster of 1, 2, 4 or 8 CTAs, every block in
// shared memory (b <= 32: eight b x b complex128 blocks a CTA), both contacts of a device in one launch.
// Products are DFMA sums in ascending k.  Near a mode threshold the iteration amplifies a rounding
// error by 1e6 and more, so these stay in FP64 arithmetic in a fixed order rather than on the tensor
// cores: any other rounding moves the self-energies there by as much as their own error.
//
// What bounds it is GB300's FP64 pipe (two DFMA a cycle and SM): six products and an elimination of
// 16 x 16 blocks are 115,000 DFMA a sweep, 57,000 cycles on one SM.  Few energies leave SMs idle, so a cluster
// splits the products' rows (each CTA writes its rows into every CTA's copy through distributed shared
// memory; two cluster barriers a sweep) while every CTA eliminates for itself.  In the elimination one
// warp finds the pivot and forms its reciprocal one step ahead, and the rows update from one copy of the block
// into another.  Contacts of b = 16 with 4 energies: 2 x 2.5 ms with a CTA each, one after the other; 0.88 ms so.
#include <cooperative_groups.h>

#include "gj64.cuh"
#include "kernels.cuh"

namespace qtx {

namespace {

namespace cg = cooperative_groups;
constexpr int kThreads = 256;

struct Lead {
  const cx<double>*H00, *H01;
  cx<double>* SR;  // [ne][n][n]
};
struct DecimArgs {
  Lead lead[2];
  const double* E;
  double eta, tol_rel;
  int max_iter, n;
  int* status;
};

template <int NM>
struct DSmem {
  static constexpr int LD = NM + 1;  // odd stride: row and column reads free of bank conflicts
  cx<double> m[8][NM * LD];
  cx<double> rowk[NM], recip;
  int perm[NM], from[NM];
  int piv;
  unsigned hi;
  double red[kThreads / 32];
};

// One entry of the update: x - f a with a the scaled pivot row, its roundings written out.
__device__ __forceinline__ cx<double> upd(cx<double> x, cx<double> f, cx<double> a) {
  return mk<double>(__dsub_rn(x.re, __fma_rn(f.re, a.re, -__dmul_rn(f.im, a.im))),
                    __dsub_rn(x.im, __fma_rn(f.im, a.re, __dmul_rn(f.re, a.im))));
}
// ... of the pivot column, 0 - f r with r = 1 / pivot: the two products' roles exchanged
__device__ __forceinline__ cx<double> upd_col(cx<double> f, cx<double> r) {
  return mk<double>(__dsub_rn(0.0, __fma_rn(-f.im, r.im, __dmul_rn(f.re, r.re))),
                    __dsub_rn(0.0, __fma_rn(f.re, r.im, __dmul_rn(f.im, r.re))));
}

// Gauss-Jordan inverse with partial (row) pivoting on |re| + |im|, first maximum on ties, from block A
// (destroyed) with B as the other copy; the result is the returned block (A or B), nullptr (uniformly)
// for a zero pivot.  Step k's chain -- the column's update, its pivot and the reciprocal (two divisions of
// 520 cycles) -- runs in warp 0 while the other warps make step k - 1's update of the remaining columns.
template <int NM>
__device__ cx<double>* eliminate(DSmem<NM>& s, cx<double>* A, cx<double>* B, const gj::FastDiv& fd) {
  constexpr int LD = DSmem<NM>::LD;
  const int t = threadIdx.x, n = fd.n;
  // the update's threads: warps 1 to 7, or while the chain decides (n <= 24) those of the other quarters of the SM,
  // each with an FP64 pipe of its own (warps 0 and 4 share one)
  const bool apart = n <= 24;
  const int kUpd = apart ? 192 : 224, u = t < 32 ? -1 : (apart ? (t < 128 ? t - 32 : (t < 160 ? kUpd * 64 : t - 64)) : t - 32);
  // pivot row of column k of block X and the reciprocal of its entry (warp 0)
  auto pivot = [&](const cx<double>* X, int k) {
    const unsigned long long key = (t >= k && t < n) ? gj::pivot_key(X[t * LD + k]) : 0ull;
    const unsigned long long best = gj::warp_max(key);
    const int p = best ? __ffs((int)__ballot_sync(0xffffffffu, key == best)) - 1 : -1;
    cx<double> r = mk<double>(0.0, 0.0);
    if (p >= 0) r = gj::crecip_warp(X[p * LD + k]);
    if (t == 0) {
      s.piv = p;
      s.perm[k] = p;
      s.recip = r;
    }
  };
  if (t < 32) pivot(A, 0);
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    const int p = s.piv;
    if (p < 0) return nullptr;
    const cx<double> r = s.recip;
    if (t < n) {  // the pivot row scaled
      const cx<double> x = A[p * LD + t];
      const cx<double> y = mk<double>(__fma_rn(x.re, r.re, -__dmul_rn(x.im, r.im)), __fma_rn(x.re, r.im, __dmul_rn(x.im, r.re)));
      s.rowk[t] = t == k ? r : y;
    }
    __syncthreads();
    // rows k and p interchanged: row i of the update comes from row src
    auto src = [&](int i) { return i == p ? k : i; };
    const int c1 = k + 1;
    if (t < 32) {
      if (c1 < n) {
        if (t < n) B[t * LD + c1] = t == k ? s.rowk[c1] : upd(A[src(t) * LD + c1], A[src(t) * LD + k], s.rowk[c1]);
        __syncwarp();
        pivot(B, c1);
      }
    } else {
      for (int idx = u; idx < n * n; idx += kUpd) {
        const int i = fd.div(idx), j = idx - i * n;
        if (j != k && j != c1) B[i * LD + j] = i == k ? s.rowk[j] : upd(A[src(i) * LD + j], A[src(i) * LD + k], s.rowk[j]);
      }
      if (t >= kThreads - 32) {
        const int i = t - (kThreads - 32);
        if (i < n) B[i * LD + k] = i == k ? s.rowk[k] : upd_col(A[src(i) * LD + k], s.rowk[k]);
      }
    }
    __syncthreads();
    cx<double>* x = A;
    A = B;
    B = x;
  }
  // the row interchanges undone as column interchanges, k = n - 1 .. 0: where result column j comes from
  if (t < n) {
    int c = t;
    for (int k = 0; k < n; ++k) {
      const int p = s.perm[k];
      c = c == k ? p : (c == p ? k : c);
    }
    s.from[t] = c;
  }
  __syncthreads();
  for (int idx = t; idx < n * n; idx += kThreads) {
    const int i = fd.div(idx), j = idx - i * n;
    B[i * LD + j] = A[i * LD + s.from[j]];
  }
  __syncthreads();
  return B;
}

// largest modulus over the n x n blocks X and Y (all threads get it)
template <int NM>
__device__ double max_mod(DSmem<NM>& s, const cx<double>* X, const cx<double>* Y, int n) {
  constexpr int LD = DSmem<NM>::LD;
  double m = 0.0;
  for (int idx = threadIdx.x; idx < n * n; idx += kThreads) {
    const cx<double> x = X[(idx / n) * LD + idx % n], y = Y[(idx / n) * LD + idx % n];
    m = fmax(m, fmax(hypot(x.re, x.im), hypot(y.re, y.im)));
  }
  for (int off = 16; off > 0; off >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, off));
  if (threadIdx.x % 32 == 0) s.red[threadIdx.x / 32] = m;
  __syncthreads();
  double r = s.red[0];
  for (int w = 1; w < kThreads / 32; ++w) r = fmax(r, s.red[w]);
  __syncthreads();
  return r;
}
// whether that modulus is below tol (tol < 2^500): the largest |re|, |im| decides by its high word unless it
// lies within sqrt(2) of tol
template <int NM>
__device__ bool below(DSmem<NM>& s, const cx<double>* X, const cx<double>* Y, int n, double tol) {
  constexpr int LD = DSmem<NM>::LD;
  unsigned h = 0;
  auto hw = [](double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; };
  for (int idx = threadIdx.x; idx < n * n; idx += kThreads) {
    const cx<double> x = X[(idx / n) * LD + idx % n], y = Y[(idx / n) * LD + idx % n];
    h = max(h, max(max(hw(x.re), hw(x.im)), max(hw(y.re), hw(y.im))));
  }
  h = __reduce_max_sync(0xffffffffu, h);
  if (threadIdx.x == 0) s.hi = 0;
  __syncthreads();
  if (threadIdx.x % 32 == 0) atomicMax(&s.hi, h);
  __syncthreads();
  h = s.hi;
  __syncthreads();
  if (h < 0x7ff00000u) {  // NaN: fmax skips it, so the exact maximum decides
    if (__hiloint2double((int)h, 0) >= tol) return false;
    if (__hiloint2double((int)h + 1, 0) * 1.4142135623731 < tol) return true;
  }
  return max_mod<NM>(s, X, Y, n) < tol;
}

template <int NM>
__device__ __forceinline__ cx<double> dot(const cx<double>* A, const cx<double>* B, int r, int c, int n) {
  constexpr int LD = DSmem<NM>::LD;
  cx<double> acc = mk<double>(0.0, 0.0);
  for (int k = 0; k < n; ++k) cfma(acc, A[r * LD + k], B[k * LD + c]);
  return acc;
}

// A contact's failure into its energy's status: of two failing contacts the first one's code stands, whichever
// cluster ends first.  Out of line: inlined, it changes the code of the
// sweeps (4 energies at b = 16: 1394 -> 1403 us a solve).
__device__ __noinline__ void raise_status(int* status, int st) {
  if (blockIdx.y == 0 && gridDim.y > 1) atomicExch(status, st);
  else atomicCAS(status, 0, st);
}

template <int NM>
__global__ void __launch_bounds__(kThreads) k_decimate(const DecimArgs a) {
  extern __shared__ __align__(16) unsigned char dsm[];
  DSmem<NM>& s = *reinterpret_cast<DSmem<NM>*>(dsm);
  constexpr int LD = DSmem<NM>::LD;
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const Lead& L = a.lead[blockIdx.y];
  const int e = blockIdx.x / C, n = a.n, t = threadIdx.x;
  const gj::FastDiv fd(n);
  // this CTA's rows of the products
  const int r0 = rank * n / C, rows = (rank + 1) * n / C - r0;
  cx<double>*al = s.m[0], *be = s.m[1], *ep = s.m[2], *es = s.m[3], *G = s.m[4], *T = s.m[5], *AG = s.m[6], *BG = s.m[7];
  const cx<double> z = mk<double>(a.E[e], a.eta);
  auto sync = [&]() {
    if (C > 1) cl.sync();
    else __syncthreads();
  };
  // v at (r, c) of block D in every CTA of the cluster
  auto put = [&](cx<double>* D, int r, int c, cx<double> v) {
    if (C == 1) {
      D[r * LD + c] = v;
      return;
    }
    for (int q = 0; q < C; ++q) *cl.map_shared_rank(&D[r * LD + c], q) = v;
  };
  for (int idx = t; idx < n * n; idx += kThreads) {
    const int r = idx / n, c = idx % n;
    al[r * LD + c] = L.H01[idx];
    be[r * LD + c] = conj(L.H01[(long)c * n + r]);
    ep[r * LD + c] = L.H00[idx];
    es[r * LD + c] = L.H00[idx];
  }
  sync();  // from here on a CTA may write into another's copies
  // tolerance relative to the coupling's largest modulus (al holds H01, be its adjoint)
  const double scale = max_mod<NM>(s, al, al, n);
  const double tol = a.tol_rel * (scale > 0.0 ? scale : 1.0);
  auto shifted = [&](const cx<double>* X) {  // AG = z - X
    for (int idx = t; idx < n * n; idx += kThreads) {
      const int r = idx / n, c = idx % n;
      const cx<double> x = X[r * LD + c];
      AG[r * LD + c] = mk<double>((r == c ? z.re : 0.0) - x.re, (r == c ? z.im : 0.0) - x.im);
    }
    __syncthreads();
  };
  bool converged = false, singular = false;
  for (int it = 1; it <= a.max_iter; ++it) {
    shifted(ep);
    cx<double>* g = eliminate<NM>(s, AG, BG, fd);
    if (!g) {
      singular = true;
      break;
    }
    // g moves to G: AG and BG take the products
    for (int idx = t; idx < n * n; idx += kThreads) G[(idx / n) * LD + idx % n] = g[(idx / n) * LD + idx % n];
    sync();  // also: every CTA is done with its AG, BG
    for (int idx = t; idx < 2 * rows * n; idx += kThreads) {
      const int w = idx >= rows * n, o = idx - w * rows * n, r = r0 + fd.div(o), c = o - fd.div(o) * n;
      put(w ? BG : AG, r, c, dot<NM>(w ? be : al, G, r, c, n));  // alpha g, beta g
    }
    sync();
    // every CTA has its G copy free now: alpha' -> G, beta' -> T; eps, eps_s in place (owned rows)
    for (int idx = t; idx < 3 * rows * n; idx += kThreads) {
      const int w = idx >= 2 * rows * n ? 2 : idx >= rows * n, o = idx - w * rows * n, r = r0 + fd.div(o), c = o - fd.div(o) * n;
      if (w == 0) {
        const cx<double> x = dot<NM>(AG, be, r, c, n);             // alpha g beta
        const cx<double> y = dot<NM>(BG, al, r, c, n);             // beta g alpha
        es[r * LD + c] = es[r * LD + c] + x;
        put(ep, r, c, (ep[r * LD + c] + x) + y);
      } else {
        put(w == 1 ? G : T, r, c, dot<NM>(w == 1 ? AG : BG, w == 1 ? al : be, r, c, n));
      }
    }
    sync();
    cx<double>* x = al;
    al = G;
    G = x;
    x = be;
    be = T;
    T = x;
    if (below<NM>(s, al, be, n, tol)) {
      converged = true;
      break;
    }
  }
  int st = 0;
  if (singular) st = (int)QTX_ERR_SINGULAR;
  else if (!converged) st = (int)QTX_ERR_NOT_CONVERGED;
  // every CTA's rows of eps_s to the first, which finishes alone
  if (C > 1) {
    if (rank)
      for (int idx = t; idx < rows * n; idx += kThreads) {
        const int r = r0 + idx / n, c = idx % n;
        *cl.map_shared_rank(&es[r * LD + c], 0) = es[r * LD + c];
      }
    cl.sync();
    if (rank) return;
  }
  cx<double>* out = L.SR + (long)e * n * n;
  // g_s = (z - eps_s)^-1 (also after a capped iteration, as the launched path does)
  cx<double>* g = nullptr;
  if (!singular) {
    shifted(es);
    for (int idx = t; idx < n * n; idx += kThreads) {
      const int r = idx / n, c = idx % n;
      al[r * LD + c] = L.H01[idx];
      be[r * LD + c] = conj(L.H01[(long)c * n + r]);
    }
    __syncthreads();
    g = eliminate<NM>(s, AG, BG, fd);
    if (!g) singular = true;
  }
  if (singular) {
    st = (int)QTX_ERR_SINGULAR;
    for (int idx = t; idx < n * n; idx += kThreads) out[idx] = mk<double>(0.0, 0.0);
  } else {
    for (int idx = t; idx < n * n; idx += kThreads) T[(idx / n) * LD + idx % n] = dot<NM>(al, g, idx / n, idx % n, n);  // H01 g_s
    __syncthreads();
    for (int idx = t; idx < n * n; idx += kThreads) out[idx] = dot<NM>(T, be, idx / n, idx % n, n);  // (H01 g_s) H01^H
  }
  if (t == 0 && st && a.status) raise_status(a.status + e, st);
}

template <int NM>
cudaError_t launch(const DecimArgs& a, int batch, int leads, cudaStream_t st) {
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = allow_smem(k_decimate<NM>, (int)sizeof(DSmem<NM>), done);
  if (e != cudaSuccess) return e;
  // CTAs of a cluster: as many as leave every energy and contact resident at once on the SMs
  int C = 1;
  while (C < 8 && (long)batch * leads * C * 2 <= kSms && 4 * C <= a.n) C *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(batch * C, leads);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = sizeof(DSmem<NM>);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if ((e = cudaLaunchKernelEx(&cfg, k_decimate<NM>, a)) != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace

cudaError_t decimate_small(int leads, const cx<double>* const* H00, const cx<double>* const* H01, cx<double>* const* SR,
                           const double* E, double eta, double tol_rel, int max_iter, int n, int batch, int* status,
                           cudaStream_t st) {
  if (n < 1 || n > kDecimSmallMax || leads < 1 || leads > 2) return cudaErrorInvalidValue;
  DecimArgs a;
  for (int k = 0; k < 2; ++k) a.lead[k] = Lead{H00[k < leads ? k : 0], H01[k < leads ? k : 0], SR[k < leads ? k : 0]};
  a.E = E; a.eta = eta; a.tol_rel = tol_rel; a.max_iter = max_iter; a.n = n; a.status = status;
  return n <= 16 ? launch<16>(a, batch, leads, st) : launch<32>(a, batch, leads, st);
}

}  // namespace qtx
