// The FP64 selected inversion of devices with small blocks (b <= 32): the whole recursion of one energy
// in one CTA, with the block products and inverses of small_block.cuh.
//
// What bounds such a device on the launched path is neither memory nor arithmetic but the chain of
// about 25 dependent launches per slice (4 to 85 us each: a 16 x 16 block fills a CTA, and its FP64
// arithmetic a sixteenth of a warp's lanes per issue on GB300's narrow FP64 pipe).  Here a slice is some
// 13 products of under a microsecond and one inverse, with the left-connected blocks of the slice and the
// full blocks of its neighbour in shared memory; g_i, g^<_i, V_i g_i and V_i g^<_i go to the plan's
// workspace between the sweeps, as on the launched path.  Formulas: see solve_chunk (rgf.cu), with
//     T = P (X2 - (P G^<_{i+1,i+1})^H / 2),   G^<_ii = g^<_i + T - T^H      (P = g_i U_i, X2 = G_{i+1,i+1} Q)
// for its two products P G^< P^H and P X2, which needs only that G^<_{i+1,i+1} is anti-Hermitian.
#include "kernels.cuh"
#include "small_block.cuh"

namespace qtx {

namespace {

using blk::kThreads;
using blk::Smem;

template <int NM>
__global__ void __launch_bounds__(kThreads) k_rgf_small(const SmallArgs a) {
  extern __shared__ __align__(16) unsigned char dsm[];
  Smem<NM>& s = *reinterpret_cast<Smem<NM>*>(dsm);
  constexpr int LD = Smem<NM>::LD;
  const int e = blockIdx.x, b = a.b, nb = a.nb;
  const long bb = (long)b * b;
  cx<double>*G = s.m[0], *GL = s.m[1], *B1 = s.m[2], *B2 = s.m[3], *P = s.m[4], *T1 = s.m[5], *T2 = s.m[6], *T3 = s.m[7];
  const double Er = a.E[e], ei = a.eta;
  const cx<double> zero = mk<double>(0.0, 0.0);
  auto slot = [&](cx<double>* base, int i) { return base + (long)i * a.slot + (long)e * bb; };
  auto out = [&](cx<double>* base, int n, int i) { return base + ((long)e * n + i) * bb; };
  auto lead = [&](const cx<double>* p) { return p + (long)e * bb; };
  // U = z S_{i,i+1} - H_{i,i+1} and V = z S^H - H^H (V may be null); zero beyond b
  auto couplings = [&](cx<double>* U, cx<double>* V, int i) {
    const cx<double>* H = a.Hu + (long)i * bb;
    const cx<double>* S = a.Su ? a.Su + (long)i * bb : nullptr;
    for (int k = threadIdx.x; k < NM * NM; k += kThreads) {
      const int r = k / NM, c = k % NM;
      const bool in = r < b && c < b;
      if (U) {
        const cx<double> h = in ? H[r * b + c] : zero;
        cx<double> v = mk<double>(-h.re, -h.im);
        if (S && in) {
          const cx<double> x = S[r * b + c];
          v = mk<double>(Er * x.re - ei * x.im - h.re, Er * x.im + ei * x.re - h.im);
        }
        U[r * LD + c] = v;
      }
      if (V) {
        const cx<double> h = in ? H[c * b + r] : zero;
        cx<double> v = mk<double>(-h.re, h.im);
        if (S && in) {
          const cx<double> x = S[c * b + r];
          v = mk<double>(Er * x.re + ei * x.im - h.re, -Er * x.im + ei * x.re + h.im);
        }
        V[r * LD + c] = v;
      }
    }
  };

  // ---- forward sweep
  for (int i = 0; i < nb; ++i) {
    const bool cL = a.SR_L && i == 0, cR = a.SR_L && i == nb - 1;
    for (int k = threadIdx.x; k < NM * NM; k += kThreads) {
      const int r = k / NM, c = k % NM;
      cx<double> v = zero;
      if (r < b && c < b) {
        const long at = (long)r * b + c;
        if (a.Sd) {
          const cx<double> x = a.Sd[(long)i * bb + at];
          v = mk<double>(Er * x.re - ei * x.im, Er * x.im + ei * x.re);
        } else if (r == c) {
          v = mk<double>(Er, ei);
        }
        v = v - a.Hd[(long)i * bb + at];
        if (a.SRd) v = v - a.SRd[(long)e * a.sSig + (long)i * bb + at];
        if (cL) v = v - lead(a.SR_L)[at];
        if (cR) v = v - lead(a.SR_R)[at];
      }
      B1[r * LD + c] = v;
    }
    cx<double>* V = P;
    if (i > 0) couplings(B2, V, i - 1);
    __syncthreads();
    if (i > 0) {
      blk::mm<NM>(s, b, T1, 1.0, V, OP_N, G, OP_N, nullptr, 0.0, true, true);   // Z = V g
      blk::store_block<NM>(slot(a.z, i - 1), T1, b);
      blk::mm<NM>(s, b, B1, -1.0, T1, OP_N, B2, OP_N, B1, 0.0, true, true);     // A - Z U
    }
    if (!blk::inverse<NM>(s, G, B1, T1, T2, b) && threadIdx.x == 0) atomicCAS(a.status + e, 0, (int)QTX_ERR_SINGULAR);
    __syncthreads();
    for (int k = threadIdx.x; k < NM * NM; k += kThreads) {
      const int r = k / NM, c = k % NM;
      cx<double> v = zero;
      if (r < b && c < b) {
        const long at = (long)r * b + c;
        if (a.SLd) v = a.SLd[(long)e * a.sSig + (long)i * bb + at];
        if (cL) v = v + lead(a.SL_L)[at];
        if (cR) v = v + lead(a.SL_R)[at];
      }
      B1[r * LD + c] = v;
    }
    __syncthreads();
    if (i > 0) {
      blk::mm<NM>(s, b, T1, 1.0, V, OP_N, GL, OP_N, nullptr, 0.0, true, true);  // X = V g^<
      blk::store_block<NM>(slot(a.x, i - 1), T1, b);
      blk::mm<NM>(s, b, B1, 1.0, T1, OP_N, V, OP_C, B1, 0.0, true, true);       // Sigma^< + X V^H
    }
    blk::mm<NM>(s, b, T1, 1.0, G, OP_N, B1, OP_N, nullptr, 0.0, true, true);
    blk::mm<NM>(s, b, GL, 1.0, T1, OP_N, G, OP_C, nullptr, 0.0, true, true);    // g^< = (g Sigma) g^H
    if (i + 1 < nb) {
      blk::store_block<NM>(slot(a.g, i), G, b);
      blk::store_block<NM>(slot(a.gl, i), GL, b);
    }
  }

  // blocks of slice i out; its density (and `cur`, the trace of interface (i, i+1)) reduced
  auto finish = [&](int i, double cur) {
    if (a.GR_diag) blk::store_block<NM>(out(a.GR_diag, nb, i), G, b);
    if (a.GL_diag) blk::store_block<NM>(out(a.GL_diag, nb, i), GL, b);
    if (a.GG_diag) {
      cx<double>* o = out(a.GG_diag, nb, i);
      blk::each<NM>(b, [&](int r, int c) {
        o[r * b + c] = GL[r * LD + c] + (G[r * LD + c] - conj(G[c * LD + r]));
      });
    }
    double den = (int)threadIdx.x < b ? GL[threadIdx.x * LD + threadIdx.x].im : 0.0;
    blk::sum2<NM>(s, cur, den);
    if (threadIdx.x == 0) {
      if (i + 1 < nb) a.cur[(long)e * a.ldcur + i] = -2.0 * cur;
      a.den[(long)e * nb + i] = den;
    }
    __syncthreads();
  };
  // Re Tr[Sigma^< G^> - Sigma^> G^<] of a contact on the present blocks, G^> = G^< + G - G^H
  auto contact_current = [&](const cx<double>* SL, const cx<double>* SG) {
    double t = 0.0, u = 0.0;
    blk::each<NM>(b, [&](int j, int k) {
      const cx<double> x = lead(SL)[j * b + k], y = lead(SG)[j * b + k], gl = GL[k * LD + j];
      const cx<double> gg = gl + (G[k * LD + j] - conj(G[j * LD + k]));
      t += (x.re * gg.re - x.im * gg.im) - (y.re * gl.re - y.im * gl.im);
    });
    blk::sum2<NM>(s, t, u);
    return t;
  };
  finish(nb - 1, 0.0);
  if (a.SR_L) {
    const double t = contact_current(a.SL_R, a.SG_R);
    if (threadIdx.x == 0) a.con[(long)e * 2 + 1] = t;
    __syncthreads();
  }

  // ---- backward sweep
  for (int i = nb - 2; i >= 0; --i) {
    blk::load_block<NM>(B1, slot(a.g, i), b);
    couplings(B2, nullptr, i);
    __syncthreads();
    blk::mm<NM>(s, b, P, 1.0, B1, OP_N, B2, OP_N, nullptr, 0.0, true, true);
    blk::load_block<NM>(B2, slot(a.z, i), b);
    __syncthreads();
    blk::mm<NM>(s, b, T1, -1.0, G, OP_N, B2, OP_N, nullptr, 0.0, true, true);   // G_{i+1,i}
    if (a.GR_lower) blk::store_block<NM>(out(a.GR_lower, nb - 1, i), T1, b);
    blk::load_block<NM>(B2, slot(a.x, i), b);
    __syncthreads();
    blk::mm<NM>(s, b, T2, 1.0, G, OP_N, B2, OP_N, nullptr, 0.0, false, true);   // X2 = G_{i+1,i+1} Q
    const bool upper = a.GR_upper || a.GG_upper;
    if (upper) {
      blk::mm<NM>(s, b, B2, -1.0, P, OP_N, G, OP_N, nullptr, 0.0, true, true);  // G_{i,i+1}
      if (a.GR_upper) blk::store_block<NM>(out(a.GR_upper, nb - 1, i), B2, b);
    }
    blk::mm<NM>(s, b, T3, 1.0, P, OP_N, GL, OP_N, nullptr, 0.0, !upper, true);  // P G^<_{i+1,i+1}
    // T3 <- G^<_{i,i+1} = -P G^< + X2^H, then T2 <- X2 - (P G^<)^H / 2 = (X2 + (G^<_{i,i+1})^H) / 2
    double cur = 0.0;
    const cx<double>* Hu = a.Hu + (long)i * bb;
    const cx<double>* Su = a.Su ? a.Su + (long)i * bb : nullptr;
    blk::each<NM>(b, [&](int r, int c) {
      const cx<double> v = conj(T2[c * LD + r]) - T3[r * LD + c];
      T3[r * LD + c] = v;
      cx<double> h = Hu[r * b + c];
      if (Su) h = h - Er * Su[r * b + c];
      cur += h.re * v.re + h.im * v.im;
      if (a.GL_upper) out(a.GL_upper, nb - 1, i)[r * b + c] = v;
      if (a.GG_upper) out(a.GG_upper, nb - 1, i)[r * b + c] = v + (B2[r * LD + c] - conj(T1[c * LD + r]));
    });
    __syncthreads();
    blk::each<NM>(b, [&](int r, int c) {
      const cx<double> v = T2[r * LD + c] + conj(T3[c * LD + r]);
      T2[r * LD + c] = mk<double>(0.5 * v.re, 0.5 * v.im);
    });
    blk::mm<NM>(s, b, G, -1.0, P, OP_N, T1, OP_N, B1, 0.0, false, true);        // G_ii = g_i - P G_{i+1,i}
    blk::mm<NM>(s, b, T1, 1.0, P, OP_N, T2, OP_N, nullptr, 0.0, false, true);
    const cx<double>* gl = slot(a.gl, i);
    blk::each<NM>(b, [&](int r, int c) { GL[r * LD + c] = gl[r * b + c] + (T1[r * LD + c] - conj(T1[c * LD + r])); });
    __syncthreads();
    finish(i, cur);
  }

  // ---- left contact: current, and T = Tr[Gam A_00] - Tr[Gam G Gam G^H] with A = i (G - G^H)
  if (a.SR_L) {
    const double t = contact_current(a.SL_L, a.SG_L);
    __syncthreads();
    blk::load_block<NM>(B1, lead(a.Gam_L), b);
    __syncthreads();
    blk::mm<NM>(s, b, T1, 1.0, B1, OP_N, G, OP_N, nullptr, 0.0, true, true);
    blk::mm<NM>(s, b, T2, 1.0, G, OP_N, B1, OP_N, nullptr, 0.0, true, true);
    double im = 0.0, fr = 0.0;
    blk::each<NM>(b, [&](int j, int k) {
      const cx<double> x = B1[j * LD + k], d = G[k * LD + j] - conj(G[j * LD + k]);
      im += x.re * d.im + x.im * d.re;
      const cx<double> p = T1[j * LD + k], q = T2[j * LD + k];
      fr += p.re * q.re + p.im * q.im;
    });
    blk::sum2<NM>(s, im, fr);
    if (threadIdx.x == 0) {
      a.con[(long)e * 2] = t;
      a.tra[e] = -im - fr;
    }
  }
}

template <int NM>
cudaError_t launch(const SmallArgs& a, int batch, cudaStream_t st) {
  static std::atomic<unsigned long long> done{0};
  const cudaError_t e = allow_smem(k_rgf_small<NM>, (int)sizeof(Smem<NM>), done);
  if (e != cudaSuccess) return e;
  k_rgf_small<NM><<<batch, kThreads, sizeof(Smem<NM>), st>>>(a);
  count_launch();
  return cudaGetLastError();
}

}  // namespace

cudaError_t rgf_small(const SmallArgs& a, int batch, cudaStream_t st) {
  if (a.b < 1 || a.b > kSmallMax) return cudaErrorInvalidValue;
  return a.b <= 16 ? launch<16>(a, batch, st) : launch<32>(a, batch, st);
}

}  // namespace qtx
