// Host orchestration and C ABI of the RGF selected inversion (declared in include/qtx_rgf.h).
//
// Per chunk of energies (all kernels batched over the chunk, one stream):
//   1. contacts: Sancho-Rubio decimation in FP64 -> Sigma^R_L,R, Gamma, Sigma^<, Sigma^>
//   2. forward sweep i = 0..N_B-1:  g_i = (A_i - V_{i-1} g_{i-1} U_{i-1})^-1,
//                                   g^<_i = g_i (Sigma^<_i + V_{i-1} g^<_{i-1} V_{i-1}^H) g_i^H
//   3. backward sweep i = N_B-2..0 for G^R, G^< blocks (formulas at `backward`), G^> = G^< + G^R - G^A
//   4. FP64 observables and their energy integrals.
// The sweep is the block Gaussian elimination of the paper's Sec. IV-A applied to Eq. 2 (Table I,
// G-row); the block inverse is a recursive 2 x 2 Schur-complement inversion over leaf blocks of at
// most 64 that are inverted with partial pivoting.  Elimination without pivoting between blocks is
// safe here for the same reason it is safe between slices: the anti-Hermitian part of M,
// eta S + Gamma/2, is positive definite, so every leading principal block and every Schur
// complement is nonsingular.
#include <algorithm>
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <thread>
#include <type_traits>
#include <vector>

#include "../../include/qtx_kernels.h"
#include "kernels.cuh"

using namespace qtx;

namespace {
thread_local std::string g_create_error;

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Byte-offset allocator for the single workspace allocation.
struct Arena {
  size_t off = 0;
  size_t take(size_t bytes) {
    const size_t o = off;
    off = align_up(off + bytes, 256);
    return o;
  }
};

// FP64 products of at least kTcF64Min in every dimension run on the tensor cores (tc_fp64.cu)
constexpr int kTcF64Min = 33;
// FP64 block inverses that do not converge by refinement are eliminated with pivots over the whole column
// up to this size (as leaves, or in global memory), by the recursion above it
constexpr int kPivotedMax = 256;

// products launched together at most (those of a slice's stage)
constexpr int kMany = 4;

// U_i, V_i differ per energy when z multiplies an overlap block or Sigma^R_{i,i+1} depends on E.
inline bool uv_per_energy(const qtx_rgf_desc& d) {
  return d.has_S || d.system_input || (d.offdiag_sigma && d.energy_dependent_sigma);
}

struct Layout {
  size_t g, gl, gl2, zk, xk, gfx, glfx, fx_slot, sig_stage, opnd[2], opnd_bytes[2], refine_act, tmp, inv_tmp, U, V, ident, ident_df, shared_blk, ref, f32a, f32tmp, dec, dec_flags, lead, obs, flags, dscale, bal, bscale, bgn, bhn, cres, cflag,
      tc_scratch, total;
  int n_tmp, n_dec;
  size_t tc_bytes;
  size_t tc_more;  // scratch of further products launched together with one in tc_scratch (n_more of them)
  int n_more;
  bool short_launches;  // a product has at most four tiles per SM (make_layout, launch_after)
  bool refine64;  // FP64 block inverses by refinement (inverse_f64) have their areas
};
}  // namespace

struct qtx_rgf_group_s;

struct qtx_rgf_plan_s {
  qtx_rgf_desc d{};
  qtx_rgf_group_s* group = nullptr;  // set while the plan solves as a member of a group
  int member = -1;
  int b = 0, nb = 0, Ec = 0;
  long bb = 0;
  size_t esz = 0;  // bytes per complex element of the sweep workspace
  Layout L{};
  unsigned char* ws = nullptr;
  std::string err;
  cudaStream_t last = nullptr;
  int* d_err_flag = nullptr;    // tensor-core engine wait/limit flag
  int worst = 0;                // worst per-energy status after the last synchronising call
  int* h_status = nullptr;      // pinned host copy of the chunk status
  int* h_flag = nullptr;        // pinned host copy of the chunk's escalation flags
  std::vector<int> status_host;
  const int* out_status = nullptr;  // caller's per-energy status array of the last solve
  int out_status_n = 0;
  // GEMM profiling (qtx_rgf_set_profiling): event pairs around each product-kernel launch
  bool prof = false;
  std::vector<cudaEvent_t> ev_pool;
  size_t ev_used = 0;
  double pipe_flops = 0.0, useful_flops = 0.0;
  cudaEvent_t* next_events() {
    if (ev_used + 2 > ev_pool.size()) {
      for (int k = 0; k < 256; ++k) {
        cudaEvent_t e;
        if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
        ev_pool.push_back(e);
      }
    }
    cudaEvent_t* r = &ev_pool[ev_used];
    ev_used += 2;
    return r;
  }
};

namespace {

// Whether a device's two contacts are iterated in the same launches: their elimination is then a leaf, one CTA
// (or cluster) a block that leaves SMs idle and lasts as long for two contacts as for one (b = 48, 12 energies:
// 20.6 -> 13.9 ms a solve).  Larger blocks run one contact after the other through one contact's buffers.
// (2 x 32767 entries: a grid's y and z extents.)
bool contacts_together(const qtx_rgf_desc& d, bool single) {
  return d.leads && !single && d.block_size <= kLeafMax && d.max_energies_in_flight <= 32767;
}

// inverse_only: the areas a batched inverse on its own uses (block g, and the refinement's), or with leads a contact
// on its own
Layout make_layout(const qtx_rgf_desc& d, bool inverse_only = false) {
  Layout L{};
  const long b = d.block_size, nb = d.n_blocks, Ec = d.max_energies_in_flight;
  const size_t bb = (size_t)b * b;
  // FP32 plans that escalate energies to FP64 lay out complex128 blocks (the FP64 re-solve runs on
  // the same workspace); df32 blocks are complex128-sized anyway
  const size_t es = (d.precision == QTX_FP32 && !(d.escalate_tol > 0)) ? sizeof(cx<float>) : sizeof(cx<double>);
  Arena a;
  // 12, 13: Sigma^<_{i,i+1} in the sweep's type and g_i Sigma^<_{i,i+1}; 14: g_i B2_{i,i+1} (second_rhs)
  L.n_tmp = inverse_only ? 0 : (d.offdiag_sigma ? (d.second_rhs ? 15 : 14) : 12);
  if (d.storage_bits) {
    // two working blocks per kind in the sweep's type (slices i and i-1 / i+1), every slice's
    // left-connected blocks in FPX: a slot of fx_slot bytes per slice and kind
    L.g = a.take(2 * Ec * bb * es);
    L.gl = a.take(2 * Ec * bb * es);
    L.fx_slot = fpx_bytes(d.storage_bits, 2 * Ec * bb);
    L.gfx = a.take(nb * L.fx_slot);
    L.glfx = a.take(nb * L.fx_slot);
  } else {
    L.g = a.take(nb * Ec * bb * es);
    L.gl = a.take(inverse_only ? 0 : nb * Ec * bb * es);
  }
  L.gl2 = a.take(d.second_rhs ? nb * Ec * bb * es : 0);  // left-connected blocks of the second right-hand side
  // Z_i = V_i g_i of every slice but the last, formed in the forward sweep and kept for the
  // backward one (without FPX storage, whose point is to keep fewer full blocks)
  L.zk = a.take(!d.storage_bits && nb > 1 ? (nb - 1) * Ec * bb * es : 0);
  // and X_i = V_i g^<_i of every right-hand side, the backward sweep's Q_i
  L.xk = a.take(!d.storage_bits && nb > 1 ? (size_t)(d.second_rhs ? 2 : 1) * (nb - 1) * Ec * bb * es : 0);
  L.tmp = a.take((size_t)L.n_tmp * Ec * bb * es);
  L.sig_stage = a.take(d.sigma_stream ? 2 * Ec * bb * sizeof(cx<double>) : 0);  // Sigma^R_ii, Sigma^<_ii
  // (the contacts' elimination recurses in complex128 whatever the sweep's type)
  L.inv_tmp = a.take(Ec * bb * (d.leads && b > kLeafMax ? sizeof(cx<double>) : es) + 4096);
  const size_t ou = uv_per_energy(d) ? (size_t)(nb > 1 ? nb - 1 : 0) * Ec * bb * es : (size_t)(nb > 1 ? nb - 1 : 0) * bb * es;
  L.U = a.take(ou);
  L.V = a.take(ou);
  // one block shared by every energy (the slice's -(H + Sigma^R) or Sigma^<, converted once)
  L.shared_blk = a.take(d.precision == QTX_FP64 ? 0 : bb * sizeof(cx<double>));
  const bool mixed = d.precision == QTX_EMU64 || d.precision == QTX_BF16X3;
  // (a contact on its own takes neither: its products and inverses stay with DFMA in a fixed order)
  const bool tc64 = d.precision == QTX_FP64 && b >= kTcF64Min && !(inverse_only && d.leads);
  L.refine64 = mixed || tc64;
  L.ident = a.take(L.refine64 ? bb * sizeof(cx<double>) : 0);
  L.ident_df = a.take(L.refine64 ? bb * sizeof(cx<double>) : 0);
  L.ref = a.take((L.refine64 || b > kLeafMax) ? 3 * Ec * bb * sizeof(cx<double>) : 0);
  L.f32a = a.take(L.refine64 ? Ec * bb * sizeof(cx<float>) : 0);
  L.f32tmp = a.take(L.refine64 ? Ec * bb * sizeof(cx<float>) + 4096 : 0);
  L.n_dec = 10;
  const long nl = contacts_together(d, inverse_only) ? 2 : 1;  // contacts iterated in the same launches
  // (smaller lead blocks are iterated in shared memory; the transmission's four blocks remain)
  const long dec_blocks = !d.leads ? 0 : (b > kDecimSmallMax ? L.n_dec * nl : 4);
  L.dec = a.take((size_t)dec_blocks * Ec * bb * sizeof(cx<double>));
  L.dec_flags = a.take(d.leads ? 2 * nl * Ec * sizeof(int) : 0);
  L.lead = a.take(d.leads && !inverse_only ? 8 * Ec * bb * sizeof(cx<double>) : 0);
  // per-energy observables: current, density, contact(2), transmission, scratch(2)
  L.obs = a.take((size_t)Ec * (2 * nb + 8) * sizeof(double));
  L.flags = a.take((size_t)Ec * 3 * sizeof(int) + 64);
  L.dscale = a.take(64);  // device scalars (the decimation's tolerance scale)
  // continuity check: per-slice balances J [Ec][nb], residuals [Ec], escalation flags [Ec]
  const bool cont = (d.outputs & QTX_OUT_CONTINUITY) || d.escalate_tol > 0;
  L.bal = a.take(cont ? (size_t)Ec * nb * sizeof(double) : 0);
  L.bscale = a.take(cont ? (size_t)Ec * nb * sizeof(double) : 0);
  L.bgn = a.take(cont ? (size_t)Ec * nb * sizeof(double) : 0);
  L.bhn = a.take(cont ? (size_t)Ec * nb * sizeof(double) : 0);
  L.cres = a.take(cont ? (size_t)Ec * sizeof(double) : 0);
  L.cflag = a.take(cont ? (size_t)Ec * sizeof(int) + 64 : 0);
  L.refine_act = a.take((size_t)Ec * 2 * sizeof(int) + 64);  // per-energy sweep masks (ping-pong)
  L.tc_bytes = 0;
  if (mixed) L.tc_bytes = gemm_tc_scratch_bytes((int)b, (int)b, (int)b, (int)Ec, d.precision == QTX_EMU64 ? 6 : 2);
  if (d.precision == QTX_EMU64)  // the Newton correction's four-plane products
    L.tc_bytes = std::max(L.tc_bytes, gemm_tc_scratch_bytes((int)b, (int)b, (int)b, (int)Ec, 4));
  // the FP32 mode's products of 96 and more (four digit planes; the recursive inverse's halves too)
  if (d.precision == QTX_FP32 && b >= 96 && b <= 1024) L.tc_bytes = gemm_tc_scratch_bytes((int)b, (int)b, (int)b, (int)Ec, 4);
  // (FP64: digit planes of up to kMany products while they are small, see gemm_fp64_tc_scratch_bytes)
  if (tc64) L.tc_bytes = gemm_fp64_tc_scratch_bytes((int)b, (int)b, (int)b, (int)(inverse_only ? Ec : kMany * Ec));
  L.tc_scratch = a.take(L.tc_bytes);
  // products of a slice that do not depend on each other share launches while one alone has at most
  // four tiles per SM (608): their further scratch is then a few hundred MB at most, and the
  // launch's tail, its fixed costs and idle SMs are paid once (b = 120, 24 energies: 72 tiles a product
  // on 152 SMs).  Larger products fill their waves alone.  Early launches of everything (launch_after) follow the same
  // count.  FP64 is counted in 64 columns too, though its tiles have 32: between four and eight waves of those, early
  // launches take 16.5 against 17.0 ms at b = 64, 23.2 against 23.7 at 100, 14.9 against 15.0 at 128 and 22.4 against 21.7
  // at 256 (310, 200, 160 and 40 energies).
  const long col = d.precision == QTX_EMU64 ? 48 : 64;
  const long tiles = ((b + 127) / 128) * ((b + col - 1) / col) * Ec;
  L.short_launches = tiles <= 4 * kSms;
  L.n_more = !inverse_only && L.tc_bytes && d.precision != QTX_FP64 && tiles <= 4 * kSms ? kMany - 1 : 0;
  L.tc_more = a.take((size_t)L.n_more * align_up(L.tc_bytes, 1024));
  // kept digitised operands (emulated modes): two left operands, b x b, E_c energies (none when the
  // products are split along K)
  for (int k = 0; k < 2; ++k) {
    L.opnd_bytes[k] = mixed ? gemm_tc_operand_bytes((int)b, (int)b, (int)Ec, d.precision == QTX_EMU64 ? 6 : 2) : 0;
    L.opnd[k] = a.take(L.opnd_bytes[k]);
  }
  L.total = a.off;
  return L;
}

const char* cuda_msg(cudaError_t e) { return cudaGetErrorString(e); }

#define QTX_CK(call)                                                      \
  do {                                                                    \
    cudaError_t e_ = (call);                                              \
    if (e_ != cudaSuccess) {                                              \
      P->err = std::string(#call) + ": " + cuda_msg(e_);                  \
      return QTX_ERR_CUDA;                                                \
    }                                                                     \
  } while (0)

// ----------------------------------------------------------------------------- solver context
template <typename T>
struct Ctx {
  qtx_rgf_plan_s* P;
  cudaStream_t st;
  int ne;                 // energies in this chunk
  const double* E;        // device energies of this chunk
  int* status;            // device status of this chunk [ne]
  long bb;
  int b;

  cx<T>* blk(size_t base, long i) const {
    return reinterpret_cast<cx<T>*>(P->ws + base) + (size_t)i * P->Ec * bb;
  }
  cx<T>* tmp(int k) const { return blk(P->L.tmp, k); }
  // left-connected / full blocks of slice i: slot i, or with FPX storage working block i % 2
  cx<T>* g(int i) const { return blk(P->L.g, P->d.storage_bits ? i % 2 : i); }
  cx<T>* gl(int i) const { return blk(P->L.gl, P->d.storage_bits ? i % 2 : i); }
  // lesser-type blocks of right-hand side k (k = 1: second_rhs, never FPX-stored)
  cx<T>* glk(int k, int i) const { return k ? blk(P->L.gl2, i) : gl(i); }
  // Z_i = V_i g_i kept from the forward sweep (nullptr without: FPX storage or one slice)
  bool keep_z() const { return !P->d.storage_bits && P->nb > 1; }
  cx<T>* zk(int i) const { return blk(P->L.zk, i); }
  // X_i = V_i g^<_i of right-hand side k, kept from the forward sweep as the backward sweep's Q_i
  cx<T>* xk(int k, int i) const { return blk(P->L.xk, (long)k * (P->nb - 1) + i); }
  void* gfx(int i) const { return P->ws + P->L.gfx + (size_t)i * P->L.fx_slot; }
  void* glfx(int i) const { return P->ws + P->L.glfx + (size_t)i * P->L.fx_slot; }
};

template <typename T>
GemmArgs<T> gargs(int M, int N, int K, const cx<T>* A, long lda, long sA, int opA, const cx<T>* B,
                  long ldb, long sB, int opB, const cx<T>* C0, long ldc0, long sC0, cx<T>* C, long ldc,
                  long sC, double alpha, double beta, int batch, const int* active) {
  GemmArgs<T> g;
  g.M = M; g.N = N; g.K = K;
  g.A = A; g.lda = lda; g.sA = sA; g.opA = opA;
  g.B = B; g.ldb = ldb; g.sB = sB; g.opB = opB;
  g.C0 = C0; g.ldc0 = ldc0; g.sC0 = sC0;
  g.C = C; g.ldc = ldc; g.sC = sC;
  g.alpha = alpha; g.beta = beta; g.batch = batch; g.active = active;
  return g;
}

// GEMM dispatch by the plan's precision (FP32 and FP64: SIMT; EMU64 / BF16X3: tensor-core engine).
// Which kept digitised left operand (tensor-core modes) a product uses: slot 0 or 1, mode KEEP (digitise into
// the slot) or REUSE (take the slot's planes: the operand, its op and its shape are unchanged since the KEEP
// product).  Ignored by the other modes.
enum { DG_NONE = 0, DG_KEEP = 1, DG_REUSE = 2 };
struct DigitHint {
  int a_slot = -1, a_mode = DG_NONE;
  int digits = 0;  // digit planes of a tensor-core product (0: the plan's)
};
inline DigitHint keepA(int slot) { DigitHint h; h.a_slot = slot; h.a_mode = DG_KEEP; return h; }
inline DigitHint reuseA(int slot) { DigitHint h; h.a_slot = slot; h.a_mode = DG_REUSE; return h; }
inline DigitHint planes(int digits) { DigitHint h; h.digits = digits; return h; }

template <typename T>
qtx_status gemm(qtx_rgf_plan_s* P, const GemmArgs<T>& g, cudaStream_t st, bool force_simt = false,
                DigitHint hint = DigitHint{});

// A tensor-core product of a plan that solves as a group member: posted to the group, launched
// together with the other members' products (defined with the group below).
cudaError_t group_gemm(qtx_rgf_plan_s* P, const TcArgs& a, int digits, cudaStream_t st);

// The profiled product kernel is the plan's own: the SIMT GEMM in the FP64 / FP32 modes, the
// tensor-core GEMM in the emulated modes (whose FP32 starting-guess inverse also calls GEMMs -- SIMT,
// or the tensor cores' four-plane FP32 instance -- which are not counted).
template <typename T>
qtx_status gemm_simt_prof(qtx_rgf_plan_s* P, const GemmArgs<T>& g, cudaStream_t st) {
  const bool mine = P->d.precision == (std::is_same<T, double>::value ? QTX_FP64 : QTX_FP32);
  cudaEvent_t* ev = (P->prof && mine) ? P->next_events() : nullptr;
  if (ev) cudaEventRecord(ev[0], st);
  QTX_CK(gemm_simt<T>(g, st));
  if (ev) {
    cudaEventRecord(ev[1], st);
    const double f = 8.0 * g.M * g.N * g.K * g.batch;
    P->pipe_flops += f;
    P->useful_flops += f;
  }
  return QTX_OK;
}
// complex64 products (the FP32 mode, and the emulated-FP64 mode's FP32 starting inverse): those of
// at least kTcF32Min in every dimension run on the tensor cores with four digit planes (~27-bit
// products, at least FP32's precision; every digit group exact), the smaller ones on the SIMT GEMM.
constexpr int kTcF32Min = 96;
inline bool f32_on_tc(const qtx_rgf_desc& d) { return d.precision != QTX_BF16X3; }
bool f32_takes_tc(qtx_rgf_plan_s* P, const GemmArgs<float>& g) {
  return f32_on_tc(P->d) && g.M >= kTcF32Min && g.N >= kTcF32Min && g.K >= kTcF32Min && g.K <= 1024 &&
         gemm_tc_scratch_bytes(g.M, g.N, g.K, g.batch, 4) <= P->L.tc_bytes;
}
inline int tc_digits(const qtx_rgf_desc& d) { return d.precision == QTX_EMU64 ? 6 : 2; }
template <typename T>
TcArgs tc_args(qtx_rgf_plan_s* P, const GemmArgs<T>& g) {
  TcArgs a;
  if (std::is_same<T, float>::value) a.ta = a.tb = a.tc = EL_F32;
  if (g.b64) a.tb = EL_F64;
  a.M = g.M; a.N = g.N; a.K = g.K;
  a.A = reinterpret_cast<const cx<df>*>(g.A); a.lda = g.lda; a.sA = g.sA; a.opA = g.opA;
  a.B = reinterpret_cast<const cx<df>*>(g.B); a.ldb = g.ldb; a.sB = g.sB; a.opB = g.opB;
  a.C0 = reinterpret_cast<const cx<df>*>(g.C0); a.ldc0 = g.ldc0; a.sC0 = g.sC0;
  a.C = reinterpret_cast<cx<df>*>(g.C); a.ldc = g.ldc; a.sC = g.sC;
  a.alpha = g.alpha; a.beta = g.beta;
  a.batch = g.batch; a.active = g.active;
  a.stages = P->d.tc_stages; a.ctas = P->d.tc_ctas;
  return a;
}
template <>
qtx_status gemm<float>(qtx_rgf_plan_s* P, const GemmArgs<float>& g, cudaStream_t st, bool, DigitHint) {
  if (f32_takes_tc(P, g)) {
    const TcArgs a = tc_args<float>(P, g);
    // in the FP32 mode these are the plan's own products (profiled); in the other modes they
    // belong to the starting inverse (not counted)
    if (P->group && gemm_tc_variant(a, 4) >= 0) {
      QTX_CK(group_gemm(P, a, 4, st));
      return QTX_OK;
    }
    cudaEvent_t* ev = (P->prof && P->d.precision == QTX_FP32) ? P->next_events() : nullptr;
    QTX_CK(gemm_tc(a, 4, P->ws + P->L.tc_scratch, P->L.tc_bytes, P->d_err_flag, st, ev));
    if (ev) {
      const double f = 8.0 * g.M * g.N * g.K * g.batch;
      P->pipe_flops += f * tc_pairs(4);
      P->useful_flops += f;
    }
    return QTX_OK;
  }
  return gemm_simt_prof<float>(P, g, st);
}
template <>
qtx_status gemm<double>(qtx_rgf_plan_s* P, const GemmArgs<double>& g, cudaStream_t st, bool force_simt, DigitHint) {
  if (!force_simt && g.M >= kTcF64Min && g.N >= kTcF64Min && g.K >= kTcF64Min && gemm_fp64_tc_fits(g.M, g.N, g.K, P->L.tc_bytes)) {
    cudaEvent_t* ev = (P->prof && P->d.precision == QTX_FP64) ? P->next_events() : nullptr;
    QTX_CK(gemm_fp64_tc(g, P->ws + P->L.tc_scratch, P->L.tc_bytes, P->d_err_flag, st, ev));
    if (ev) {
      const double f = 8.0 * g.M * g.N * g.K * g.batch;
      P->pipe_flops += f * tc_pairs_fp64();
      P->useful_flops += f;
    }
    return QTX_OK;
  }
  return gemm_simt_prof<double>(P, g, st);
}
// kept left operand: only for the plan's b x b x b products at the plan's digit count, when slots exist
bool kept_operand(qtx_rgf_plan_s* P, const GemmArgs<df>& g, const DigitHint& hint, int digits, TcOperand& oa) {
  const bool square = g.M == P->b && g.N == P->b && g.K == P->b && g.batch <= P->Ec && digits == tc_digits(P->d);
  if (!square || hint.a_mode == DG_NONE || !P->L.opnd_bytes[hint.a_slot]) return false;
  oa = tc_operand_at(P->ws + P->L.opnd[hint.a_slot], P->b, P->b, P->Ec, tc_digits(P->d));
  oa.mode = hint.a_mode;
  return true;
}
template <>
qtx_status gemm<df>(qtx_rgf_plan_s* P, const GemmArgs<df>& g, cudaStream_t st, bool, DigitHint hint) {
  TcArgs a = tc_args<df>(P, g);
  const int digits = hint.digits > 0 ? hint.digits : tc_digits(P->d);
  TcOperand oa;
  if (kept_operand(P, g, hint, digits, oa)) a.opndA = &oa;
  if (P->group && gemm_tc_variant(a, digits) >= 0) {
    QTX_CK(group_gemm(P, a, digits, st));
    return QTX_OK;
  }
  // the profile times the products at the plan's digit count (one kernel instance)
  cudaEvent_t* ev = (P->prof && digits == tc_digits(P->d)) ? P->next_events() : nullptr;
  QTX_CK(gemm_tc(a, digits, P->ws + P->L.tc_scratch, P->L.tc_bytes, P->d_err_flag, st, ev));
  if (ev) {
    const double f = 8.0 * g.M * g.N * g.K * g.batch;
    P->pipe_flops += f * tc_pairs(digits);
    P->useful_flops += f;
  }
  return QTX_OK;
}

// Products that do not depend on each other, issued in order.  Where the plan has scratch for several
// (Layout::n_more), up to kMany of them share one digitisation and one persistent launch; every tile is
// computed as in a launch of its own, so the results are the same bits.
bool group_pools(qtx_rgf_plan_s* P);  // the plan solves in a group that pools products
template <typename T>
struct Prods {
  GemmArgs<T> g[kTcMaxGroup];
  DigitHint h[kTcMaxGroup];
  int n = 0;
  void add(const GemmArgs<T>& x, DigitHint hint = DigitHint{}) {
    g[n] = x;
    h[n++] = hint;
  }
};
template <typename T>
qtx_status run(qtx_rgf_plan_s* P, Prods<T>& q, cudaStream_t st) {
  int i = 0;
  if constexpr (!std::is_same<T, double>::value) {
    bool many = P->L.n_more > 0 && !P->prof && !group_pools(P);
    if constexpr (std::is_same<T, float>::value)
      for (int k = 0; k < q.n; ++k) many = many && f32_takes_tc(P, q.g[k]);
    if (std::is_same<T, df>::value && P->b > 1024) many = false;  // split along K
    while (many && q.n - i > 1) {
      const int m = std::min(q.n - i, P->L.n_more + 1);
      TcArgs a[kMany];
      int digits[kMany];
      TcOperand oa[kMany];
      void* scr[kMany];
      TcPrepared p[kMany];
      const TcPrepared* pp[kMany];
      for (int k = 0; k < m; ++k) {
        a[k] = tc_args<T>(P, q.g[i + k]);
        if constexpr (std::is_same<T, float>::value) {
          digits[k] = 4;
        } else {
          digits[k] = tc_digits(P->d);
          if (kept_operand(P, q.g[i + k], q.h[i + k], digits[k], oa[k])) a[k].opndA = &oa[k];
        }
        scr[k] = k ? P->ws + P->L.tc_more + (size_t)(k - 1) * align_up(P->L.tc_bytes, 1024) : P->ws + P->L.tc_scratch;
        pp[k] = &p[k];
      }
      QTX_CK(gemm_tc_prepare_many(a, digits, m, scr, P->L.tc_bytes, P->d_err_flag, st, p));
      QTX_CK(gemm_tc_launch(pp, m, st));
      i += m;
    }
  }
  if constexpr (std::is_same<T, double>::value) {
    while (!P->prof && q.n - i > 1) {
      int m = 0;  // leading products that take the tensor cores
      while (i + m < q.n && q.g[i + m].M >= kTcF64Min && q.g[i + m].N >= kTcF64Min && q.g[i + m].K >= kTcF64Min) ++m;
      m = m > 1 ? gemm_fp64_tc_many(q.g + i, m, P->L.tc_bytes) : m;
      if (m < 2) break;
      QTX_CK(gemm_fp64_tc_launch(q.g + i, m, P->ws + P->L.tc_scratch, P->L.tc_bytes, P->d_err_flag, st));
      i += m;
    }
  }
  for (; i < q.n; ++i)
    if (const qtx_status s = gemm<T>(P, q.g[i], st, false, q.h[i])) return s;
  q.n = 0;
  return QTX_OK;
}

// Two products that do not depend on each other: one SIMT launch where both take the SIMT kernel.
template <typename T>
qtx_status gemm_pair(qtx_rgf_plan_s* P, const GemmArgs<T>& g1, const GemmArgs<T>& g2, cudaStream_t st) {
  if constexpr (std::is_same<T, float>::value) {
    if (!f32_takes_tc(P, g1) && !f32_takes_tc(P, g2) && !P->prof) {
      GemmMulti<T> m;
      m.n = 2;
      m.g[0] = g1;
      m.g[1] = g2;
      QTX_CK(gemm_simt_multi<T>(m, st));
      return QTX_OK;
    }
  }
  const qtx_status s = gemm<T>(P, g1, st, true);
  return s ? s : gemm<T>(P, g2, st, true);
}

// Plain (non-refined) recursive inverse of n x n blocks stored with leading dimension lda.
// T12/T21 scratch for each recursion level is carved from `scratch` (>= 0.7 n^2 per batch entry).
template <typename T>
qtx_status inverse_rec(qtx_rgf_plan_s* P, cx<T>* A, long lda, long sA, int n, int batch,
                       const int* active, int* status, cx<T>* scratch, long sScr, cudaStream_t st,
                       bool force_simt) {
  if (n <= kLeafMax) {
    QTX_CK(leaf_inverse<T>(A, lda, sA, n, batch, active, status, st));
    return QTX_OK;
  }
  const int h = (n + 1) / 2, r = n - h;
  cx<T>* A11 = A;
  cx<T>* A12 = A + h;
  cx<T>* A21 = A + (long)h * lda;
  cx<T>* A22 = A + (long)h * lda + h;
  cx<T>* T12 = scratch;              // h x r, ld r
  cx<T>* T21 = scratch + (long)h * r; // r x h, ld h
  cx<T>* next = scratch + 2L * h * r;
  qtx_status s;
  if ((s = inverse_rec<T>(P, A11, lda, sA, h, batch, active, status, next, sScr, st, force_simt))) return s;
  // T12 = X11 A12 ; T21 = A21 X11
  if ((s = gemm_pair<T>(P, gargs<T>(h, r, h, A11, lda, sA, OP_N, A12, lda, sA, OP_N, nullptr, 0, 0, T12, r, sScr, 1.0, 0.0, batch, active),
                        gargs<T>(r, h, h, A21, lda, sA, OP_N, A11, lda, sA, OP_N, nullptr, 0, 0, T21, h, sScr, 1.0, 0.0, batch, active), st))) return s;
  // A22 <- A22 - A21 T12 (Schur complement), then invert it in place
  if ((s = gemm<T>(P, gargs<T>(r, r, h, A21, lda, sA, OP_N, T12, r, sScr, OP_N, A22, lda, sA, A22, lda, sA, -1.0, 1.0, batch, active), st, force_simt))) return s;
  if ((s = inverse_rec<T>(P, A22, lda, sA, r, batch, active, status, next, sScr, st, force_simt))) return s;
  // A12 <- -T12 Y ; A21 <- -Y T21 ; A11 <- X11 - T12 A21
  if ((s = gemm_pair<T>(P, gargs<T>(h, r, r, T12, r, sScr, OP_N, A22, lda, sA, OP_N, nullptr, 0, 0, A12, lda, sA, -1.0, 0.0, batch, active),
                        gargs<T>(r, h, r, A22, lda, sA, OP_N, T21, h, sScr, OP_N, nullptr, 0, 0, A21, lda, sA, -1.0, 0.0, batch, active), st))) return s;
  if ((s = gemm<T>(P, gargs<T>(h, h, r, T12, r, sScr, OP_N, A21, lda, sA, OP_N, A11, lda, sA, A11, lda, sA, -1.0, 1.0, batch, active), st, force_simt))) return s;
  return QTX_OK;
}

// Recursive inverse followed, when the recursion splits the block (n > kLeafMax), by one Newton
// step X <- X + X (I - A X) in the same precision: elimination without pivoting between the two
// halves can lose digits on ill-conditioned leading blocks (e.g. the decimation's z - eps), and one
// step brings the result back to the accuracy of a pivoted inverse.
template <typename T>
qtx_status inverse_refined(qtx_rgf_plan_s* P, cx<T>* A, int n, int batch, const int* active,
                           int* status, cudaStream_t st) {
  const long nn = (long)n * n;
  cx<T>* scr = reinterpret_cast<cx<T>*>(P->ws + P->L.inv_tmp);
  if (n <= kLeafMax) return inverse_rec<T>(P, A, n, nn, n, batch, active, status, scr, nn, st, true);
  cx<T>* Acopy = reinterpret_cast<cx<T>*>(P->ws + P->L.ref);
  cx<T>* R = Acopy + (size_t)P->Ec * nn;
  cx<T>* Xn = R + (size_t)P->Ec * nn;
  Term<T> tA; tA.p = A; tA.s = nn; tA.alpha = 1.0;
  Term<T> none;
  QTX_CK((combine<T, T>(Acopy, nn, tA, none, none, n, batch, nullptr, 0.0, 0.0, active, st)));
  qtx_status s = inverse_rec<T>(P, A, n, nn, n, batch, active, status, scr, nn, st, true);
  if (s) return s;
  // R = I - Acopy X  (identity via the diagonal term of combine), Xn = X + X R, X <- Xn
  if ((s = gemm<T>(P, gargs<T>(n, n, n, Acopy, n, nn, OP_N, A, n, nn, OP_N, nullptr, 0, 0, R, n, nn, -1.0, 0.0, batch, active), st, true))) return s;
  QTX_CK(add_identity<T>(R, nn, n, batch, active, st));
  if ((s = gemm<T>(P, gargs<T>(n, n, n, A, n, nn, OP_N, R, n, nn, OP_N, A, n, nn, Xn, n, nn, 1.0, 1.0, batch, active), st, true))) return s;
  Term<T> tX; tX.p = Xn; tX.s = nn; tX.alpha = 1.0;
  QTX_CK((combine<T, T>(A, nn, tX, none, none, n, batch, nullptr, 0.0, 0.0, active, st)));
  return QTX_OK;
}

// FP32 inverse used as the emulated modes' starting guess (the df32 Newton sweeps that follow only
// need ||I - A X0|| < 1); its scratch lives in the FP32 area so the df32 buffers stay intact.
qtx_status inverse_refined_f32(qtx_rgf_plan_s* P, cx<float>* A, int n, int batch, const int* active,
                               int* status, cudaStream_t st) {
  const long nn = (long)n * n;
  cx<float>* scr = reinterpret_cast<cx<float>*>(P->ws + P->L.f32tmp);
  return inverse_rec<float>(P, A, n, nn, n, batch, active, status, scr, nn, st, true);
}

// FP64 block inverse of blocks beyond the fused leaf: X0 from the FP32 inverse, then Newton sweeps
// X <- X + X (I - A X) with FP64 products on the tensor cores, which double the correct digits each
// (an FP32 start leaves ||I - A X0|| near kappa 2^-24, so blocks of kappa 1e3 take three sweeps and
// of 1e6 five).  An energy stops after the sweep whose residual norm was at most 2^-27: the next
// residual is then its square, below FP64's resolution.  Energies still above it after kSweeps64
// (ill-conditioned beyond FP32's reach, or non-finite) are inverted again from A by pivoted
// elimination in FP64 (n = 64, 64 blocks of kappa 1e9: 0.87 ms in all, 1.40 by DFMA leaves alone).  A DFMA
// Gauss-Jordan of a 64 x 64 leaf took 770 us on one SM (GB300's FP64 pipe runs at 1/64 of its FP32 rate); the FP32
// leaf takes 37 us.  An FP64 solve of b = 128, 12 slices and 8 energies:
// 132 ms by DFMA products and leaves, 8.6 ms with products on the tensor cores and these inverses.
constexpr int kSweeps64 = 5;
qtx_status inverse_f64(qtx_rgf_plan_s* P, cx<double>* A, int n, int batch, const int* active, int* status,
                       cudaStream_t st) {
  if (n < kTcF64Min || n != P->b || !P->L.refine64 || !gemm_fp64_tc_fits(n, n, n, P->L.tc_bytes))
    return inverse_refined<double>(P, A, n, batch, active, status, st);
  const long nn = (long)n * n;
  cx<float>* A32 = reinterpret_cast<cx<float>*>(P->ws + P->L.f32a);
  cx<double>* Acopy = reinterpret_cast<cx<double>*>(P->ws + P->L.ref);
  cx<double>* R = Acopy + (size_t)P->Ec * nn;
  cx<double>* Xn = R + (size_t)P->Ec * nn;
  const cx<double>* I = reinterpret_cast<const cx<double>*>(P->ws + P->L.ident);
  Term<double> tA; tA.p = A; tA.s = nn; tA.alpha = 1.0;
  Term<double> none;
  Term<float> none32;
  QTX_CK((combine<double, float>(A32, nn, tA, none, none, n, batch, nullptr, 0.0, 0.0, active, st)));
  QTX_CK((combine<double, double>(Acopy, nn, tA, none, none, n, batch, nullptr, 0.0, 0.0, active, st)));
  qtx_status s = inverse_refined_f32(P, A32, n, batch, active, nullptr, st);
  if (s) return s;
  Term<float> tX; tX.p = A32; tX.s = nn; tX.alpha = 1.0;
  QTX_CK((combine<float, double>(A, nn, tX, none32, none32, n, batch, nullptr, 0.0, 0.0, active, st)));
  int* masks = reinterpret_cast<int*>(P->ws + P->L.refine_act);
  const int* act = active;
  for (int it = 0; it < kSweeps64; ++it) {
    int* next = masks + (it & 1) * P->Ec;
    if ((s = gemm<double>(P, gargs<double>(n, n, n, Acopy, n, nn, OP_N, A, n, nn, OP_N, I, n, 0, R, n, nn, -1.0, 1.0, batch, act), st))) return s;
    QTX_CK(residual_mask<double>(R, nn, n, batch, 0x1p-27, act, next, nullptr, st));
    // X <- X + X R, in place while the whole contraction is one launch (the product reads X through
    // its digit planes; a block with a non-finite entry races, and ends in the elimination below)
    cx<double>* dst = n <= 512 ? A : Xn;
    if ((s = gemm<double>(P, gargs<double>(n, n, n, A, n, nn, OP_N, R, n, nn, OP_N, A, n, nn, dst, n, nn, 1.0, 1.0, batch, act), st))) return s;
    if (dst == Xn) {
      Term<double> tXn; tXn.p = Xn; tXn.s = nn; tXn.alpha = 1.0;
      QTX_CK((combine<double, double>(A, nn, tXn, none, none, n, batch, nullptr, 0.0, 0.0, act, st)));
    }
    act = next;
  }
  Term<double> tC; tC.p = Acopy; tC.s = nn; tC.alpha = 1.0;
  QTX_CK((combine<double, double>(A, nn, tC, none, none, n, batch, nullptr, 0.0, 0.0, act, st)));
  if (n <= kLeafMax) {
    QTX_CK(leaf_inverse<double>(A, n, nn, n, batch, act, status, st));
    return QTX_OK;
  }
  if (n <= kPivotedMax) {
    QTX_CK(pivoted_inverse(A, nn, n, batch, act, status, st));
    return QTX_OK;
  }
  return inverse_refined<double>(P, A, n, batch, act, status, st);
}

// Block inverse used by the sweep.  FP64: inverse_f64.  FP32: recursive inverse in FP32.
// EMU64 / BF16X3: X0 from the recursive inverse in FP32, then Newton refinement
// X <- X + X (I - A X) with both products on the tensor-core engine (the residual I - A X is
// formed in emulated FP64 before it is rounded for the correction product).
template <typename T>
qtx_status block_inverse(qtx_rgf_plan_s* P, cx<T>* A, int n, int batch, const int* active,
                         int* status, cudaStream_t st);

template <>
qtx_status block_inverse<float>(qtx_rgf_plan_s* P, cx<float>* A, int n, int batch, const int* active,
                                int* status, cudaStream_t st) {
  return inverse_refined<float>(P, A, n, batch, active, status, st);
}

template <>
qtx_status block_inverse<double>(qtx_rgf_plan_s* P, cx<double>* A, int n, int batch, const int* active,
                                 int* status, cudaStream_t st) {
  return inverse_f64(P, A, n, batch, active, status, st);
}

// Emulated modes (df32 storage): X0 from the FP32 inverse of the leading parts, then Newton sweeps
// X <- X + X (I - A X) with both products on the tensor-core engine; the residual I - A X is formed
// by the engine's ~38-bit products with I added exactly in the epilogue.
template <>
qtx_status block_inverse<df>(qtx_rgf_plan_s* P, cx<df>* A, int n, int batch, const int* active,
                             int* status, cudaStream_t st) {
  const long nn = (long)n * n;
  cx<float>* A32 = reinterpret_cast<cx<float>*>(P->ws + P->L.f32a);
  cx<df>* Acopy = reinterpret_cast<cx<df>*>(P->ws + P->L.ref);
  cx<df>* R = Acopy + (size_t)P->Ec * nn;
  cx<df>* Xn = R + (size_t)P->Ec * nn;
  const cx<df>* I = reinterpret_cast<const cx<df>*>(P->ws + P->L.ident_df);
  Term<df> tA; tA.p = A; tA.s = nn; tA.alpha = 1.0;
  Term<df> none;
  QTX_CK((combine<df, float>(A32, nn, tA, none, none, n, batch, nullptr, 0.0, 0.0, active, st)));
  QTX_CK((combine<df, df>(Acopy, nn, tA, none, none, n, batch, nullptr, 0.0, 0.0, active, st)));
  qtx_status s = inverse_refined_f32(P, A32, n, batch, active, status, st);
  if (s) return s;
  Term<float> tX; tX.p = A32; tX.s = nn; tX.alpha = 1.0;
  Term<float> none32;
  QTX_CK((combine<float, df>(A, nn, tX, none32, none32, n, batch, nullptr, 0.0, 0.0, active, st)));
  // With refine_tol > 0 an energy leaves the sweeps once ||I - A X||_F <= refine_tol: the masks
  // (ping-pong in refine_act) make every later product, digitisation and combination skip it.
  int* masks = reinterpret_cast<int*>(P->ws + P->L.refine_act);
  const int* act = active;
  for (int it = 0; it < P->d.refine_max_iter; ++it) {
    // Acopy's digit planes serve every sweep
    if ((s = gemm<df>(P, gargs<df>(n, n, n, Acopy, n, nn, OP_N, A, n, nn, OP_N, I, n, 0, R, n, nn, -1.0, 1.0, batch, act), st,
                      false, it == 0 ? keepA(0) : reuseA(0)))) return s;
    int* next = nullptr;
    if (P->d.refine_tol > 0.0 && it + 1 < P->d.refine_max_iter) {
      next = masks + (it & 1) * P->Ec;
      QTX_CK(residual_mask(R, nn, n, batch, P->d.refine_tol, act, next, status, st));
    }
    // The correction X R is small (||R|| <= 2^-12 once an energy is refined, and typically near the
    // FP32 inverse's kappa 2^-24), so four digit planes (~27-bit operands, every digit group exact)
    // keep its error near 2^-27 |X| |R|, far below the 2^-40 the sweep keeps; R itself, where A X
    // cancels against I, takes the plan's six.
    const DigitHint xr = tc_digits(P->d) == 6 ? planes(4) : DigitHint{};
    if (n <= 1024) {
      // X <- X + X R in place: the product reads X only through its digit planes (made before the
      // launch) and, element by element in the epilogue, as C0 right before writing C
      if ((s = gemm<df>(P, gargs<df>(n, n, n, A, n, nn, OP_N, R, n, nn, OP_N, A, n, nn, A, n, nn, 1.0, 1.0, batch, act), st,
                        false, xr))) return s;
    } else {
      // split along K: a later K-chunk digitises columns of X an earlier chunk would have overwritten
      if ((s = gemm<df>(P, gargs<df>(n, n, n, A, n, nn, OP_N, R, n, nn, OP_N, A, n, nn, Xn, n, nn, 1.0, 1.0, batch, act), st,
                        false, xr))) return s;
      Term<df> tXn; tXn.p = Xn; tXn.s = nn; tXn.alpha = 1.0;
      QTX_CK((combine<df, df>(A, nn, tXn, none, none, n, batch, nullptr, 0.0, 0.0, act, st)));
    }
    if (next) act = next;
  }
  return QTX_OK;
}

// ----------------------------------------------------------------------------- contacts
// Batched Sancho-Rubio decimation (FP64) of one or both contacts; result Sigma^R = H01 g_s H01^H in SR.
// Nothing here reads back to the host: for lead blocks of at most kDecimSmallMax the whole iteration
// of an energy and contact runs in one cluster (decimate_small); larger blocks run decim_max_iter sweeps of
// batched launches in which converged energies are masked off on the device (their launches return at once),
// with the tolerance scale max|H01| computed on the device too.  A solve with contacts therefore
// makes no host synchronisation and can be captured in a CUDA graph.  Two contacts share the launches
// (energies of the first, then of the second) where contacts_together.
template <typename T>
qtx_status contacts(const Ctx<T>& c, int nl, const cx<double>* const* H00, const cx<double>* const* H01, double eta,
                    cx<double>* const* SR) {
  qtx_rgf_plan_s* P = c.P;
  const int b = c.b, ne = c.ne;
  const long bb = c.bb;
  cudaStream_t st = c.st;
  if (b <= kDecimSmallMax) {
    QTX_CK(decimate_small(nl, H00, H01, SR, c.E, eta, P->d.decim_tol, P->d.decim_max_iter, b, ne, c.status, st));
    return QTX_OK;
  }
  const int N = nl * ne;
  cx<double>* D = reinterpret_cast<cx<double>*>(P->ws + P->L.dec);
  auto buf = [&](int k) { return D + (size_t)k * nl * P->Ec * bb; };
  cx<double>*alpha = buf(0), *beta = buf(1), *eps = buf(2), *eps_s = buf(3), *g = buf(4), *ag = buf(5),
  *bg = buf(6), *t1 = buf(7), *t2 = buf(8), *t3 = buf(9);
  int* active = reinterpret_cast<int*>(P->ws + P->L.dec_flags);
  int* status = nl > 1 ? active + (size_t)nl * P->Ec : c.status;
  double* scale = reinterpret_cast<double*>(P->ws + P->L.dscale);

  Term<double> none;
  for (int k = 0; k < nl; ++k) {
    const size_t o = (size_t)k * ne * bb;
    QTX_CK(max_modulus(H01[k], bb, scale + k, st));
    Term<double> t01; t01.p = H01[k]; t01.s = 0; t01.alpha = 1.0;
    Term<double> t01h = t01; t01h.op = OP_C;
    Term<double> t00; t00.p = H00[k]; t00.s = 0; t00.alpha = 1.0;
    QTX_CK((combine<double, double>(alpha + o, bb, t01, none, none, b, ne, nullptr, 0, 0, nullptr, st)));
    QTX_CK((combine<double, double>(beta + o, bb, t01h, none, none, b, ne, nullptr, 0, 0, nullptr, st)));
    QTX_CK((combine<double, double>(eps + o, bb, t00, none, none, b, ne, nullptr, 0, 0, nullptr, st)));
    QTX_CK((combine<double, double>(eps_s + o, bb, t00, none, none, b, ne, nullptr, 0, 0, nullptr, st)));
    t00.alpha = -1.0;
    QTX_CK((combine<double, double>(g + o, bb, t00, none, none, b, ne, c.E, eta, 1.0, nullptr, st)));  // z - eps
  }
  QTX_CK(fill_int(active, 1, N, st));
  if (nl > 1) QTX_CK(fill_int(status, 0, N, st));
  qtx_status s;
  auto G = [&](const cx<double>* A, const cx<double>* B, cx<double>* C) {
    return gargs<double>(b, b, b, A, b, bb, OP_N, B, b, bb, OP_N, nullptr, 0, 0, C, b, bb, 1.0, 0.0, N, active);
  };
  for (int it = 1; it <= P->d.decim_max_iter; ++it) {
    // three launches a sweep beside the inverse's: a converged energy's CTAs return at once
    if ((s = inverse_refined<double>(P, g, b, N, active, status, st))) return s;
    GemmMulti<double> m;
    m.n = 2;
    m.g[0] = G(alpha, g, ag);
    m.g[1] = G(beta, g, bg);
    QTX_CK(gemm_simt_multi<double>(m, st));
    m.n = 4;
    m.g[0] = G(ag, beta, t1);   // alpha g beta
    m.g[1] = G(bg, alpha, t2);  // beta g alpha
    m.g[2] = G(ag, alpha, t3);  // alpha g alpha
    m.g[3] = G(bg, beta, g);    // beta g beta
    QTX_CK(gemm_simt_multi<double>(m, st));
    // converged energies leave stale blocks in the exchanged buffers, which nothing reads again
    std::swap(alpha, t3);
    std::swap(beta, g);
    // eps_s, eps, the convergence flags and the next sweep's z - eps (in g)
    QTX_CK(decim_update(eps_s, eps, t1, t2, alpha, beta, g, c.E, eta, ne, nl, b, P->d.decim_tol, scale, active, st));
  }
  QTX_CK(flag_active(active, status, (int)QTX_ERR_NOT_CONVERGED, N, st));
  for (int k = 0; k < nl; ++k) {
    const size_t o = (size_t)k * ne * bb;
    Term<double> tes; tes.p = eps_s + o; tes.s = bb; tes.alpha = -1.0;
    QTX_CK((combine<double, double>(g + o, bb, tes, none, none, b, ne, c.E, eta, 1.0, nullptr, st)));  // z - eps_s
  }
  if ((s = inverse_refined<double>(P, g, b, N, nullptr, status, st))) return s;
  // Sigma^R = H01 g_s H01^H
  GemmMulti<double> m;
  m.n = nl;
  for (int k = 0; k < nl; ++k)
    m.g[k] = gargs<double>(b, b, b, H01[k], b, 0, OP_N, g + (size_t)k * ne * bb, b, bb, OP_N, nullptr, 0, 0, t1 + (size_t)k * ne * bb, b,
                           bb, 1.0, 0.0, ne, nullptr);
  QTX_CK(gemm_simt_multi<double>(m, st));
  for (int k = 0; k < nl; ++k)
    m.g[k] = gargs<double>(b, b, b, t1 + (size_t)k * ne * bb, b, bb, OP_N, H01[k], b, 0, OP_C, nullptr, 0, 0, SR[k], b, bb, 1.0, 0.0, ne,
                           nullptr);
  QTX_CK(gemm_simt_multi<double>(m, st));
  if (nl > 1) QTX_CK(merge_status(status, nl, ne, c.status, st));
  return QTX_OK;
}

// Copy/convert a sweep block (batch stride bb) into a complex128 output [e][slice] layout.
template <typename T>
qtx_status emit(qtx_rgf_plan_s* P, void* out, long nslices, long slice, int e0, const cx<T>* src,
                int b, int ne, cudaStream_t st, const cx<T>* plus = nullptr, const cx<T>* minus_h = nullptr) {
  if (!out) return QTX_OK;
  const long bb = (long)b * b;
  cx<double>* o = reinterpret_cast<cx<double>*>(out) + ((long)e0 * nslices + slice) * bb;
  Term<T> t0; t0.p = src; t0.s = bb; t0.alpha = 1.0;
  Term<T> t1; t1.p = plus; t1.s = bb; t1.alpha = 1.0;
  Term<T> t2; t2.p = minus_h; t2.s = bb; t2.alpha = -1.0; t2.op = OP_C;
  QTX_CK((combine<T, double>(o, nslices * bb, t0, t1, t2, b, ne, nullptr, 0.0, 0.0, nullptr, st)));
  return QTX_OK;
}

// Per-energy observables of the chunk in the workspace.
struct ObsBufs {
  int ncur;
  double *cur, *den, *con, *tra;         // [ne][ncur], [ne][nb], [ne][2], [ne]
  double *bal, *bscale, *bgn, *bhn;      // [ne][nb] each (continuity check)
  explicit ObsBufs(qtx_rgf_plan_s* P) {
    const int nb = P->nb;
    ncur = nb > 1 ? nb - 1 : 1;
    cur = reinterpret_cast<double*>(P->ws + P->L.obs);
    den = cur + (size_t)P->Ec * ncur;
    con = den + (size_t)P->Ec * nb;
    tra = con + (size_t)P->Ec * 2;
    bal = reinterpret_cast<double*>(P->ws + P->L.bal);
    bscale = reinterpret_cast<double*>(P->ws + P->L.bscale);
    bgn = reinterpret_cast<double*>(P->ws + P->L.bgn);
    bhn = reinterpret_cast<double*>(P->ws + P->L.bhn);
  }
};
inline bool wants_balance(const qtx_rgf_desc& d) { return (d.outputs & QTX_OUT_CONTINUITY) || d.escalate_tol > 0; }

// After a chunk's sweeps: the continuity check, the per-energy outputs and the energy integrals.
template <typename T>
qtx_status finish_chunk(qtx_rgf_plan_s* P, const qtx_rgf_inputs* in, const qtx_rgf_outputs* out, int e0, int ne,
                        cudaStream_t st) {
  const qtx_rgf_desc& d = P->d;
  const int nb = P->nb;
  const unsigned m = d.outputs;
  const ObsBufs ob(P);
  const int ncur = ob.ncur;
  double *cur = ob.cur, *den = ob.den, *con = ob.con, *tra = ob.tra;
  auto want = [&](unsigned bit, const void* p) { return (m & bit) && p; };
  // ---- continuity residual per energy (and the escalation flags)
  if (wants_balance(d)) {
    double* cres = reinterpret_cast<double*>(P->ws + P->L.cres);
    int* cflag = reinterpret_cast<int*>(P->ws + P->L.cflag);
    // unit error of the products in this mode (Eq. 6: error ~ kappa eps): 6 (7) bf16 digits ~41 bits,
    // 2 digits ~13 bits, complex64 24 bits, FP64 53
    const double eps_mode = std::is_same<T, double>::value ? 0x1p-53
                            : std::is_same<T, float>::value  ? 0x1p-24
                            : (d.precision == QTX_BF16X3 ? 0x1p-13 : 0x1p-40);
    QTX_CK(continuity(cur, ncur, ob.bal, ob.bscale, ob.bgn, ob.bhn, nb, d.leads ? con : nullptr, in->energies + e0, nb, ne,
                      d.escalate_tol > 0 ? d.escalate_tol : 1e300, eps_mode, cres, cflag, st));
    if (want(QTX_OUT_CONTINUITY, out->continuity))
      QTX_CK(cudaMemcpyAsync(out->continuity + e0, cres, (size_t)ne * sizeof(double), cudaMemcpyDeviceToDevice, st));
  }
  // ---- 4. outputs of the per-energy observables and their integrals
  const int nbm1 = nb - 1;
  if (want(QTX_OUT_CURRENT, out->current) && nbm1 > 0)
    QTX_CK(cudaMemcpyAsync(out->current + (size_t)e0 * nbm1, cur, (size_t)ne * nbm1 * sizeof(double), cudaMemcpyDeviceToDevice, st));
  if (want(QTX_OUT_DENSITY, out->density))
    QTX_CK(cudaMemcpyAsync(out->density + (size_t)e0 * nb, den, (size_t)ne * nb * sizeof(double), cudaMemcpyDeviceToDevice, st));
  if (d.leads && want(QTX_OUT_CONTACT, out->contact))
    QTX_CK(cudaMemcpyAsync(out->contact + (size_t)e0 * 2, con, (size_t)ne * 2 * sizeof(double), cudaMemcpyDeviceToDevice, st));
  if (d.leads && want(QTX_OUT_TRANSMISSION, out->transmission))
    QTX_CK(cudaMemcpyAsync(out->transmission + e0, tra, (size_t)ne * sizeof(double), cudaMemcpyDeviceToDevice, st));
  if (m & QTX_OUT_INTEGRALS) {
    if (out->current_int && nbm1 > 0)
      QTX_CK(integrate_add(out->current_int, cur, nbm1, nbm1, in->weights, in->energies, e0, in->n_energies, ne, 1.0, st));
    if (out->density_int)
      QTX_CK(integrate_add(out->density_int, den, nb, nb, in->weights, in->energies, e0, in->n_energies, ne, 1.0 / (2.0 * 3.14159265358979323846), st));
  }
  return QTX_OK;
}

template <typename T>
qtx_status solve_chunk(qtx_rgf_plan_s* P, const qtx_rgf_inputs* in, const qtx_rgf_outputs* out,
                       int e0, int ne, int* status, cudaStream_t st) {
  const qtx_rgf_desc& d = P->d;
  const int b = P->b, nb = P->nb;
  const long bb = P->bb;
  Ctx<T> c{P, st, ne, in->energies + e0, status, bb, b};
  const double eta = in->eta;
  const cx<double>* Hd = reinterpret_cast<const cx<double>*>(in->H_diag);
  const cx<double>* Hu = reinterpret_cast<const cx<double>*>(in->H_upper);
  const cx<double>* Sd = d.has_S ? reinterpret_cast<const cx<double>*>(in->S_diag) : nullptr;
  const cx<double>* Su = d.has_S ? reinterpret_cast<const cx<double>*>(in->S_upper) : nullptr;
  const cx<double>* SRd = d.has_scattering ? reinterpret_cast<const cx<double>*>(in->SigR_diag) : nullptr;
  const cx<double>* SLd = d.has_scattering ? reinterpret_cast<const cx<double>*>(in->SigL_diag) : nullptr;
  const long sSig = d.energy_dependent_sigma ? (long)nb * bb : 0;
  const long sigE0 = d.energy_dependent_sigma ? (long)e0 * nb * bb : 0;
  auto sigR = [&](int i) { return SRd ? SRd + sigE0 + (long)i * bb : nullptr; };
  auto sigL = [&](int i) { return SLd ? SLd + sigE0 + (long)i * bb : nullptr; };
  // second right-hand side (second_rhs): B2 in the layout of Sigma^<
  const int nrhs = d.second_rhs ? 2 : 1;
  const cx<double>* SGd = d.second_rhs ? reinterpret_cast<const cx<double>*>(in->SigG_diag) : nullptr;
  auto sigG = [&](int i) { return SGd ? SGd + sigE0 + (long)i * bb : nullptr; };
  // off-diagonal scattering blocks [N_E or 1][N_B-1][b][b]
  const bool odg = d.offdiag_sigma && nb > 1;
  const long sSigU = d.energy_dependent_sigma ? (long)(nb - 1) * bb : 0;
  const long sigUE0 = d.energy_dependent_sigma ? (long)e0 * (nb - 1) * bb : 0;
  const cx<double>* SRu = odg && !d.system_input ? reinterpret_cast<const cx<double>*>(in->SigR_upper) + sigUE0 : nullptr;
  const cx<double>* SRl = odg && !d.system_input ? reinterpret_cast<const cx<double>*>(in->SigR_lower) + sigUE0 : nullptr;
  const cx<double>* SLu = odg ? reinterpret_cast<const cx<double>*>(in->SigL_upper) + sigUE0 : nullptr;
  const cx<double>* SGu = odg && d.second_rhs ? reinterpret_cast<const cx<double>*>(in->SigG_upper) + sigUE0 : nullptr;
  // Sigma^<_{i,i+1} in the sweep's type (tmp 12; the second right-hand side's: tmp 10): one block shared by the chunk, or one per energy
  const int nLt = d.energy_dependent_sigma ? ne : 1;
  const long sLt = d.energy_dependent_sigma ? bb : 0;
  // right-hand side k's upper block of slice i (k = 1: B2_{i,i+1})
  auto load_L = [&](int k, int i) -> cx<T>* {
    cx<T>* Lt = c.tmp(k ? 10 : 12);
    if (axpby_from64<T>(Lt, bb, (k ? SGu : SLu) + (long)i * bb, sSigU, 1.0, nullptr, 0, 0.0, b, nLt, st) != cudaSuccess) return nullptr;
    return Lt;
  };
  qtx_status s;
  Term<T> none;

  // ---- 1. contacts
  cx<double>* LB = reinterpret_cast<cx<double>*>(P->ws + P->L.lead);
  auto lb = [&](int k) { return LB + (size_t)k * P->Ec * bb; };
  cx<double>*SR_L = lb(0), *Gam_L = lb(1), *SL_L = lb(2), *SG_L = lb(3);
  cx<double>*SR_R = lb(4), *Gam_R = lb(5), *SL_R = lb(6), *SG_R = lb(7);
  if (d.leads) {
    const cx<double>* H00[2] = {(const cx<double>*)in->lead_H00_L, (const cx<double>*)in->lead_H00_R};
    const cx<double>* H01[2] = {(const cx<double>*)in->lead_H01_L, (const cx<double>*)in->lead_H01_R};
    cx<double>* SR[2] = {SR_L, SR_R};
    const int nl = contacts_together(d, false) ? 2 : 1;
    for (int k = 0; k < 2; k += nl)
      if ((s = contacts<T>(c, nl, H00 + k, H01 + k, eta, SR + k))) return s;
    QTX_CK(lead_sigmas(SR_L, Gam_L, SL_L, SG_L, c.E, in->mu_L, in->kT, b, ne, st));
    QTX_CK(lead_sigmas(SR_R, Gam_R, SL_R, SG_R, c.E, in->mu_R, in->kT, b, ne, st));
  }

  // ---- FP64 devices of small blocks: the sweeps of each energy in one CTA
  const unsigned m = d.outputs;
  auto want = [&](unsigned bit, const void* p) { return (m & bit) && p; };
  if constexpr (std::is_same<T, double>::value) {
    // the options beyond the plain sweeps (block-tridiagonal Sigma, M given, FPX storage, streamed Sigma,
    // current balances) stay on the launched path
    if (b <= kSmallMax && !d.offdiag_sigma && !d.system_input && !d.storage_bits && !d.sigma_stream && !wants_balance(d)) {
      const ObsBufs ob(P);
      SmallArgs a{};
      a.b = b; a.nb = nb;
      a.Hd = Hd; a.Hu = Hu; a.Sd = Sd; a.Su = Su; a.SRd = sigR(0); a.SLd = sigL(0);
      a.sSig = sSig;
      a.E = c.E; a.eta = eta;
      if (d.leads) {
        a.SR_L = SR_L; a.Gam_L = Gam_L; a.SL_L = SL_L; a.SG_L = SG_L;
        a.SR_R = SR_R; a.SL_R = SL_R; a.SG_R = SG_R;
      }
      a.slot = (long)P->Ec * bb;
      a.g = c.g(0); a.gl = c.gl(0);
      if (nb > 1) { a.z = c.zk(0); a.x = c.xk(0, 0); }
      auto blocks = [&](unsigned bit, void* p, long n) {
        return want(bit, p) ? reinterpret_cast<cx<double>*>(p) + (long)e0 * n * bb : nullptr;
      };
      a.GR_diag = blocks(QTX_OUT_GR_DIAG, out->GR_diag, nb);
      a.GR_upper = blocks(QTX_OUT_GR_UPPER, out->GR_upper, nb - 1);
      a.GR_lower = blocks(QTX_OUT_GR_LOWER, out->GR_lower, nb - 1);
      a.GL_diag = blocks(QTX_OUT_GL_DIAG, out->GL_diag, nb);
      a.GL_upper = blocks(QTX_OUT_GL_UPPER, out->GL_upper, nb - 1);
      a.GG_diag = blocks(QTX_OUT_GG_DIAG, out->GG_diag, nb);
      a.GG_upper = blocks(QTX_OUT_GG_UPPER, out->GG_upper, nb - 1);
      a.cur = ob.cur; a.den = ob.den; a.con = ob.con; a.tra = ob.tra;
      a.ldcur = ob.ncur;
      a.status = status;
      cudaEvent_t* ev = P->prof ? P->next_events() : nullptr;
      if (ev) cudaEventRecord(ev[0], st);
      QTX_CK(rgf_small(a, ne, st));
      if (ev) {
        cudaEventRecord(ev[1], st);
        // its products: 6 a slice (2 of the first) and 6 an interface (7 with G_{i,i+1}), 2 of the transmission
        const int n = 6 * nb - 4 + (nb - 1) * (6 + (a.GR_upper || a.GG_upper)) + (d.leads ? 2 : 0);
        const double f = 8.0 * b * b * b * n * ne;
        P->pipe_flops += f * tc_pairs_fp64();
        P->useful_flops += f;
      }
      return finish_chunk<T>(P, in, out, e0, ne, st);
    }
  }

  // ---- off-diagonal blocks of M
  cx<T>* Ub = reinterpret_cast<cx<T>*>(P->ws + P->L.U);
  cx<T>* Vb = reinterpret_cast<cx<T>*>(P->ws + P->L.V);
  const bool uvE = uv_per_energy(d);
  const long sUV = uvE ? bb : 0;
  auto U = [&](int i) { return Ub + (size_t)i * (uvE ? P->Ec * bb : bb); };
  auto V = [&](int i) { return Vb + (size_t)i * (uvE ? P->Ec * bb : bb); };
  // system input (M given): per-energy blocks [N_E][N_B(-1)][b][b]
  const cx<double>* Md = d.system_input ? reinterpret_cast<const cx<double>*>(in->M_diag) + (long)e0 * nb * bb : nullptr;
  const cx<double>* Mu = d.system_input && nb > 1 ? reinterpret_cast<const cx<double>*>(in->M_upper) + (long)e0 * (nb - 1) * bb : nullptr;
  const cx<double>* Ml = d.system_input && nb > 1 ? reinterpret_cast<const cx<double>*>(in->M_lower) + (long)e0 * (nb - 1) * bb : nullptr;
  for (int i = 0; i + 1 < nb; ++i) {
    if (d.system_input) {
      QTX_CK(axpby_from64<T>(U(i), bb, Mu + (long)i * bb, (long)(nb - 1) * bb, 1.0, nullptr, 0, 0.0, b, ne, st));
      QTX_CK(axpby_from64<T>(V(i), bb, Ml + (long)i * bb, (long)(nb - 1) * bb, 1.0, nullptr, 0, 0.0, b, ne, st));
      continue;
    }
    const cx<double>* sru = SRu ? SRu + (long)i * bb : nullptr;
    const cx<double>* srl = SRl ? SRl + (long)i * bb : nullptr;
    if (uvE) QTX_CK(assemble_offdiag<T>(U(i), V(i), Hu + (long)i * bb, Su ? Su + (long)i * bb : nullptr, c.E, eta, b, ne, st, sru, srl, sSigU));
    else QTX_CK(assemble_offdiag<T>(U(i), V(i), Hu + (long)i * bb, nullptr, nullptr, 0.0, b, 1, st, sru, srl, 0));
  }

  // products of a stage, launched together by run(); b x b blocks with batch strides sA_, sB_
  Prods<T> pr;
  auto pd = [&](const cx<T>* A, long sA_, int opA, const cx<T>* B, long sB_, int opB, const cx<T>* C0, cx<T>* C, double al, double be) {
    return gargs<T>(b, b, b, A, b, sA_, opA, B, b, sB_, opB, C0, b, bb, C, b, bb, al, be, ne, nullptr);
  };

  // ---- 2. forward sweep
  for (int i = 0; i < nb; ++i) {
    cx<T>* gi = c.g(i);
    const cx<double>* lead = nullptr;
    if (d.leads && i == 0) lead = SR_L;
    else if (d.leads && i == nb - 1) lead = SR_R;
    // streamed self-energies: this slice's blocks of the chunk's energies, host -> staging area
    const cx<double>* sRi = sigR(i);
    const cx<double>* sLi = sigL(i);
    long sS = sSig;
    if (d.sigma_stream) {
      cx<double>* stR = reinterpret_cast<cx<double>*>(P->ws + P->L.sig_stage);
      cx<double>* stL = stR + (size_t)P->Ec * bb;
      const size_t row = (size_t)bb * sizeof(cx<double>), pitch = (size_t)nb * row;
      if (pitch < ((size_t)1 << 31)) {  // one strided copy per kind
        QTX_CK(cudaMemcpy2DAsync(stR, row, sRi, pitch, row, ne, cudaMemcpyHostToDevice, st));
        QTX_CK(cudaMemcpy2DAsync(stL, row, sLi, pitch, row, ne, cudaMemcpyHostToDevice, st));
      } else {                          // pitches beyond the 2D copy's range: one copy per energy
        for (int e = 0; e < ne; ++e) {
          QTX_CK(cudaMemcpyAsync(stR + (size_t)e * bb, sRi + (size_t)e * nb * bb, row, cudaMemcpyHostToDevice, st));
          QTX_CK(cudaMemcpyAsync(stL + (size_t)e * bb, sLi + (size_t)e * nb * bb, row, cudaMemcpyHostToDevice, st));
        }
      }
      sRi = stR;
      sLi = stL;
      sS = bb;
    }
    cx<T>* shared_blk = reinterpret_cast<cx<T>*>(P->ws + P->L.shared_blk);
    if (d.system_input) QTX_CK(axpby_from64<T>(gi, bb, Md + (long)i * bb, (long)nb * bb, 1.0, nullptr, 0, 0.0, b, ne, st));
    else if (!std::is_same<T, double>::value && !Sd && (sS == 0 || !sRi) && !lead) {
      // Sigma^R shared by the energies: -(H_ii + Sigma^R_ii) converted once, then E + i eta added
      // on each energy's diagonal
      QTX_CK(axpby_from64<T>(shared_blk, 0, Hd + (long)i * bb, 0, -1.0, sRi, 0, -1.0, b, 1, st));
      QTX_CK(broadcast_diag<T>(gi, bb, shared_blk, b, c.E, eta, ne, st));
    } else QTX_CK(assemble_diag<T>(gi, Hd + (long)i * bb, Sd ? Sd + (long)i * bb : nullptr, sRi, sS, lead, bb, c.E, eta, b, ne, st));
    if (d.leads && nb == 1) {  // one slice touches both contacts
      Term<T> tg; tg.p = gi; tg.s = bb; tg.alpha = 1.0;
      QTX_CK((combine<T, T>(c.tmp(0), bb, tg, none, none, b, ne, nullptr, 0, 0, nullptr, st)));
      QTX_CK(axpby_from64<T>(c.tmp(1), bb, SR_R, bb, -1.0, nullptr, 0, 0.0, b, ne, st));
      Term<T> t0; t0.p = c.tmp(0); t0.s = bb; t0.alpha = 1.0;
      Term<T> t1; t1.p = c.tmp(1); t1.s = bb; t1.alpha = 1.0;
      QTX_CK((combine<T, T>(gi, bb, t0, t1, none, b, ne, nullptr, 0, 0, nullptr, st)));
    }
    // Sigma^<_ii (+ contacts; or B2_ii) of each right-hand side
    auto SLk = [&](int k) { return c.tmp(k ? 5 : 1); };
    for (int k = 0; k < nrhs; ++k) {
      cx<T>* SLi = SLk(k);
      const cx<double>* sl = k ? sigG(i) : sLi;
      const cx<double>* lsl = nullptr;
      if (k == 0 && d.leads && i == 0) lsl = SL_L;
      else if (k == 0 && d.leads && i == nb - 1) lsl = SL_R;
      if (sl && !lsl && sS == 0 && !std::is_same<T, double>::value) {  // shared: converted once
        QTX_CK(axpby_from64<T>(shared_blk, 0, sl, 0, 1.0, nullptr, 0, 0.0, b, 1, st));
        QTX_CK(broadcast_diag<T>(SLi, bb, shared_blk, b, nullptr, 0.0, ne, st));
      } else if (sl) QTX_CK(axpby_from64<T>(SLi, bb, sl, sS, 1.0, lsl, bb, 1.0, b, ne, st));
      else if (lsl) QTX_CK(axpby_from64<T>(SLi, bb, lsl, bb, 1.0, nullptr, 0, 0.0, b, ne, st));
      else QTX_CK(cudaMemsetAsync(SLi, 0, (size_t)ne * bb * sizeof(cx<T>), st));
      if (k == 0 && d.leads && nb == 1) {
        QTX_CK(axpby_from64<T>(c.tmp(2), bb, SL_R, bb, 1.0, nullptr, 0, 0.0, b, ne, st));
        Term<T> t0; t0.p = SLi; t0.s = bb; t0.alpha = 1.0;
        Term<T> t1; t1.p = c.tmp(2); t1.s = bb; t1.alpha = 1.0;
        QTX_CK((combine<T, T>(SLi, bb, t0, t1, none, b, ne, nullptr, 0, 0, nullptr, st)));
      }
    }
    if (i > 0) {
      const bool kz = c.keep_z();
      // Z = V g and X = V g^<, kept for the backward sweep (G_{i,i-1} = -G_ii Z and Q = X); V g U is then
      // Z U.  Without them V (g U), where g_{i-1} was the left operand of the previous slice's g Sigma^< and
      // its digit planes are kept
      cx<T>* Zf = kz ? c.zk(i - 1) : c.tmp(2);
      cx<T>* gU = c.tmp(0);
      auto Xk = [&](int k) { return kz ? c.xk(k, i - 1) : c.tmp(4); };
      if (kz || odg) pr.add(pd(V(i - 1), sUV, OP_N, c.g(i - 1), bb, OP_N, nullptr, Zf, 1.0, 0.0));
      if (!kz) pr.add(pd(c.g(i - 1), bb, OP_N, U(i - 1), sUV, OP_N, nullptr, gU, 1.0, 0.0), reuseA(1));
      for (int k = 0; k < nrhs; ++k) pr.add(pd(V(i - 1), sUV, OP_N, c.glk(k, i - 1), bb, OP_N, nullptr, Xk(k), 1.0, 0.0));
      if ((s = run<T>(P, pr, st))) return s;
      if (kz) pr.add(pd(Zf, bb, OP_N, U(i - 1), sUV, OP_N, gi, gi, -1.0, 1.0));
      else pr.add(pd(V(i - 1), sUV, OP_N, gU, bb, OP_N, gi, gi, -1.0, 1.0));
      for (int k = 0; k < nrhs; ++k) pr.add(pd(Xk(k), bb, OP_N, V(i - 1), sUV, OP_C, SLk(k), SLk(k), 1.0, 1.0));
      auto Yf = [&](int k) { return c.tmp(k ? 6 : 3); };
      if (odg)  // block-tridiagonal Sigma^<: bracket += -Y + Y^H, Y = V_{i-1} g_{i-1} Sigma^<_{i-1,i}
        for (int k = 0; k < nrhs; ++k) {
          cx<T>* Lt = load_L(k, i - 1);
          if (!Lt) return QTX_ERR_CUDA;
          pr.add(pd(Zf, bb, OP_N, Lt, sLt, OP_N, nullptr, Yf(k), 1.0, 0.0));
        }
      if ((s = run<T>(P, pr, st))) return s;
      if (odg)
        for (int k = 0; k < nrhs; ++k) {
          Term<T> t0; t0.p = SLk(k); t0.s = bb; t0.alpha = 1.0;
          Term<T> t1; t1.p = Yf(k); t1.s = bb; t1.alpha = -1.0;
          Term<T> t2; t2.p = Yf(k); t2.s = bb; t2.alpha = 1.0; t2.op = OP_C;
          QTX_CK((combine<T, T>(SLk(k), bb, t0, t1, t2, b, ne, nullptr, 0, 0, nullptr, st)));
        }
    }
    if ((s = block_inverse<T>(P, gi, b, ne, nullptr, status, st))) return s;
    // left-connected lesser functions g Sigma g^H
    auto Yk = [&](int k) { return c.tmp(k ? 6 : 0); };
    for (int k = 0; k < nrhs; ++k) pr.add(pd(gi, bb, OP_N, SLk(k), bb, OP_N, nullptr, Yk(k), 1.0, 0.0), k ? reuseA(1) : keepA(1));
    if ((s = run<T>(P, pr, st))) return s;
    for (int k = 0; k < nrhs; ++k) pr.add(pd(Yk(k), bb, OP_N, gi, bb, OP_C, nullptr, c.glk(k, i), 1.0, 0.0));
    if ((s = run<T>(P, pr, st))) return s;
    // FPX storage: slices the backward sweep reads back from memory (the last two stay in the
    // working blocks) are kept compressed
    if (d.storage_bits && i < nb - 2) {
      QTX_CK(fpx_store<T>(d.storage_bits, gi, (long)ne * bb, c.gfx(i), st));
      QTX_CK(fpx_store<T>(d.storage_bits, c.gl(i), (long)ne * bb, c.glfx(i), st));
    }
  }

  // ---- 3. backward sweep.  With P = g_i U_i, Z = V_i g_i, Q = V_i g^<_i:
  //   G_{i+1,i} = -G_{i+1,i+1} Z,  G_{i,i+1} = -P G_{i+1,i+1},  G_ii = g_i - P G_{i+1,i}
  //   X2 = G_{i+1,i+1} Q   (block-tridiagonal Sigma^<: Q += (g_i Sigma^<_{i,i+1})^H)
  //   G^<_{i,i+1} = -P G^<_{i+1,i+1} + X2^H     [= -P G^< - g^< V^H G^A]
  //   G^<_ii = g^<_i + T - T^H,  T = P (X2 - (P G^<_{i+1,i+1})^H / 2)
  // The last line is g^<_i + P G^<_{i+1,i+1} P^H + P X2 - (P X2)^H with G^<_{i+1,i+1} anti-Hermitian: its
  // congruence is (Y - Y^H) / 2 with Y = -P (P G^<)^H, so one product P (..) serves both terms: 12 products a
  // slice (13 with G_{i,i+1}) instead of 14, and the current's error against 64 bits falls to a third.
  const ObsBufs ob(P);
  const int ncur = ob.ncur;
  double *cur = ob.cur, *den = ob.den, *con = ob.con, *tra = ob.tra;
  // current conservation (Sec. II-B): per-slice balances J_i, checked after the sweep
  const bool cont = wants_balance(d);
  double *bal = ob.bal, *bscale = ob.bscale, *bgn = ob.bgn, *bhn = ob.bhn;
  double* spare = tra;  // the second right-hand side's traces, which nothing reads (no contacts then)
  {
    const int i = nb - 1;
    if (want(QTX_OUT_GR_DIAG, out->GR_diag) && (s = emit<T>(P, out->GR_diag, nb, i, e0, c.g(i), b, ne, st))) return s;
    if (want(QTX_OUT_GL_DIAG, out->GL_diag) && (s = emit<T>(P, out->GL_diag, nb, i, e0, c.gl(i), b, ne, st))) return s;
    if (want(QTX_OUT_GG_DIAG, out->GG_diag) &&
        (s = d.second_rhs ? emit<T>(P, out->GG_diag, nb, i, e0, c.glk(1, i), b, ne, st)
                          : emit<T>(P, out->GG_diag, nb, i, e0, c.gl(i), b, ne, st, c.g(i), c.g(i))))
      return s;
    QTX_CK(obs_density<T>(den + i, nb, c.gl(i), bb, b, ne, st));
    if (cont)
      QTX_CK(obs_balance<T>(bal + i, bscale + i, bgn + i, bhn + i, nb, sigL(i), sigR(i), sSig, c.g(i), c.gl(i), bb,
                            eta, b, ne, st, Hd + (long)i * bb, nullptr, nullptr, c.E, nullptr));
    if (d.leads) {  // right contact current on slice N_B-1:  G^> = G^< + G^R - G^A
      cx<T>* GG = c.tmp(0);
      Term<T> t0; t0.p = c.gl(i); t0.s = bb; t0.alpha = 1.0;
      Term<T> t1; t1.p = c.g(i); t1.s = bb; t1.alpha = 1.0;
      Term<T> t2; t2.p = c.g(i); t2.s = bb; t2.alpha = -1.0; t2.op = OP_C;
      QTX_CK((combine<T, T>(GG, bb, t0, t1, t2, b, ne, nullptr, 0, 0, nullptr, st)));
      QTX_CK(obs_trace2<T>(con + 1, 2, SL_R, bb, GG, bb, SG_R, bb, c.gl(i), bb, b, ne, st));
    }
  }
  for (int i = nb - 2; i >= 0; --i) {
    const bool kz = c.keep_z();
    cx<T>* GRn = c.g(i + 1);
    cx<T>* Pm = c.tmp(2);
    cx<T>* Z = kz ? c.zk(i) : c.tmp(3);  // V_i g_i
    cx<T>* GRl = c.tmp(4);
    cx<T>* GRu = c.tmp(5);
    cx<T>* GLu = c.tmp(10);
    cx<T>* gi = c.g(i);
    // per right-hand side (the second one comes with kept Z and X only)
    auto Qk = [&](int k) { return kz ? c.xk(k, i) : c.tmp(6); };  // V_i g^<_i: the forward sweep's X when kept
    auto X2k = [&](int k) { return c.tmp(k ? 3 : 9); };
    auto PGLk = [&](int k) { return c.tmp(k ? 11 : 8); };
    auto Tk = [&](int k) { return c.tmp(k ? 6 : 7); };
    auto Rl = [&](int k) { return c.tmp(13 + k); };               // g_i L_k with L_k its upper block
    if (d.storage_bits && i < nb - 2) {  // g_i, g^<_i back from FPX into the working blocks
      QTX_CK(fpx_load<T>(d.storage_bits, c.gfx(i), (long)ne * bb, gi, st));
      QTX_CK(fpx_load<T>(d.storage_bits, c.glfx(i), (long)ne * bb, c.gl(i), st));
    }
    // kept digit planes (tensor-core modes): slot 0 = P (left operand of three or four products), slot 1 =
    // G_{i+1,i+1} (left operand of two)
    pr.add(pd(gi, bb, OP_N, U(i), sUV, OP_N, nullptr, Pm, 1.0, 0.0));
    if (!kz) {
      pr.add(pd(V(i), sUV, OP_N, gi, bb, OP_N, nullptr, Z, 1.0, 0.0));
      pr.add(pd(V(i), sUV, OP_N, c.gl(i), bb, OP_N, nullptr, Qk(0), 1.0, 0.0));
    }
    if (odg)
      for (int k = 0; k < nrhs; ++k) {  // g_i still left-connected
        cx<T>* Lt = load_L(k, i);
        if (!Lt) return QTX_ERR_CUDA;
        pr.add(pd(gi, bb, OP_N, Lt, sLt, OP_N, nullptr, Rl(k), 1.0, 0.0));
      }
    if ((s = run<T>(P, pr, st))) return s;
    if (odg)
      for (int k = 0; k < nrhs; ++k) {  // Q = V_i g^<_i + (g_i Sigma^<_{i,i+1})^H
        Term<T> t0; t0.p = Qk(k); t0.s = bb; t0.alpha = 1.0;
        Term<T> t1; t1.p = Rl(k); t1.s = bb; t1.alpha = 1.0; t1.op = OP_C;
        QTX_CK((combine<T, T>(Qk(k), bb, t0, t1, none, b, ne, nullptr, 0, 0, nullptr, st)));
      }
    // G_{i,i+1} only where it is an output (itself, or in G^>_{i,i+1}) or the balance check's K needs it
    const bool want_u = want(QTX_OUT_GR_UPPER, out->GR_upper) || (!d.second_rhs && want(QTX_OUT_GG_UPPER, out->GG_upper)) || cont;
    pr.add(pd(GRn, bb, OP_N, Z, bb, OP_N, nullptr, GRl, -1.0, 0.0), keepA(1));
    for (int k = 0; k < nrhs; ++k) pr.add(pd(GRn, bb, OP_N, Qk(k), bb, OP_N, nullptr, X2k(k), 1.0, 0.0), reuseA(1));
    for (int k = 0; k < nrhs; ++k) pr.add(pd(Pm, bb, OP_N, c.glk(k, i + 1), bb, OP_N, nullptr, PGLk(k), 1.0, 0.0), k ? reuseA(0) : keepA(0));
    if (want_u) pr.add(pd(Pm, bb, OP_N, GRn, bb, OP_N, nullptr, GRu, -1.0, 0.0), reuseA(0));
    if ((s = run<T>(P, pr, st))) return s;
    if (want(QTX_OUT_GR_UPPER, out->GR_upper) && (s = emit<T>(P, out->GR_upper, nb - 1, i, e0, GRu, b, ne, st))) return s;
    if (want(QTX_OUT_GR_LOWER, out->GR_lower) && (s = emit<T>(P, out->GR_lower, nb - 1, i, e0, GRl, b, ne, st))) return s;
    // G^<_{i,i+1}, written where an output or the balance reads it, with its current trace; X2 becomes the
    // right operand of T
    void* traces = c.tmp(0);  // (tmp 0 and 1: lesser_scratch_bytes exceeds one block for b = 1)
    const bool cur_out = !d.system_input;
    for (int k = 0; k < nrhs; ++k) {
      const bool gg = !d.second_rhs && want(QTX_OUT_GG_UPPER, out->GG_upper);
      const bool up = k ? want(QTX_OUT_GG_UPPER, out->GG_upper) : want(QTX_OUT_GL_UPPER, out->GL_upper) || gg || cont;
      const bool ck = k == 0 && cur_out;
      QTX_CK(lesser_offdiag<T>(PGLk(k), X2k(k), up ? GLu : nullptr, ck ? Hu + (long)i * bb : nullptr,
                               ck && Su ? Su + (long)i * bb : nullptr, c.E, b, ne, traces, st));
      if (k == 1) {  // the second right-hand side's blocks are the GG outputs
        if (up && (s = emit<T>(P, out->GG_upper, nb - 1, i, e0, GLu, b, ne, st))) return s;
        continue;
      }
      if (want(QTX_OUT_GL_UPPER, out->GL_upper) && (s = emit<T>(P, out->GL_upper, nb - 1, i, e0, GLu, b, ne, st))) return s;
      if (gg && (s = emit<T>(P, out->GG_upper, nb - 1, i, e0, GLu, b, ne, st, GRu, GRl))) return s;
    }
    pr.add(pd(Pm, bb, OP_N, GRl, bb, OP_N, gi, gi, -1.0, 1.0), reuseA(0));   // g_i <- G_ii
    if (cont) {
      // plans that check the current balance form K and the congruence apart: T - T^H is anti-Hermitian
      // whatever the rounding, so the balance would no longer see the part of it that the check measures
      pr.add(pd(GRu, bb, OP_N, Qk(0), bb, OP_N, nullptr, Tk(0), -1.0, 0.0));
      pr.add(pd(PGLk(0), bb, OP_N, Pm, bb, OP_C, c.gl(i), c.gl(i), 1.0, 1.0));
    } else {
      for (int k = 0; k < nrhs; ++k) pr.add(pd(Pm, bb, OP_N, X2k(k), bb, OP_N, nullptr, Tk(k), 1.0, 0.0), reuseA(0));
    }
    if ((s = run<T>(P, pr, st))) return s;
    if (want(QTX_OUT_GR_DIAG, out->GR_diag) && (s = emit<T>(P, out->GR_diag, nb, i, e0, gi, b, ne, st))) return s;
    for (int k = 0; k < nrhs; ++k) {
      cx<T>* gli = c.glk(k, i);
      const long o64 = ((long)e0 * nb + i) * bb;
      void* gd = k ? (want(QTX_OUT_GG_DIAG, out->GG_diag) ? out->GG_diag : nullptr)
                   : (want(QTX_OUT_GL_DIAG, out->GL_diag) ? out->GL_diag : nullptr);
      QTX_CK(lesser_diag<T>(gli, Tk(k), gd ? reinterpret_cast<cx<double>*>(gd) + o64 : nullptr, (long)nb * bb,
                            k == 0 && cur_out ? cur + i : nullptr, ncur, Su != nullptr, k ? spare : den + i, k ? 1 : nb, b, ne, traces, st));   // G^<_ii
      if (k == 1) continue;
      if (!d.second_rhs && want(QTX_OUT_GG_DIAG, out->GG_diag) && (s = emit<T>(P, out->GG_diag, nb, i, e0, gli, b, ne, st, gi, gi))) return s;
      if (cont)
        QTX_CK(obs_balance<T>(bal + i, bscale + i, bgn + i, bhn + i, nb, sigL(i), sigR(i), sSig, gi, gli, bb, eta, b,
                              ne, st, Hd + (long)i * bb, Hu + (long)i * bb, Su ? Su + (long)i * bb : nullptr, c.E, GLu));
    }
  }
  if (d.leads) {  // left contact current and transmission on slice 0
    cx<T>* GG = c.tmp(0);
    Term<T> t0; t0.p = c.gl(0); t0.s = bb; t0.alpha = 1.0;
    Term<T> t1; t1.p = c.g(0); t1.s = bb; t1.alpha = 1.0;
    Term<T> t2; t2.p = c.g(0); t2.s = bb; t2.alpha = -1.0; t2.op = OP_C;
    QTX_CK((combine<T, T>(GG, bb, t0, t1, t2, b, ne, nullptr, 0, 0, nullptr, st)));
    QTX_CK(obs_trace2<T>(con, 2, SL_L, bb, GG, bb, SG_L, bb, c.gl(0), bb, b, ne, st));
    // T = Tr[Gam A_00] - Tr[Gam G Gam G^H] with A = i (G - G^H): Tr[Gam A] = -Im Tr[Gam (G - G^H)],
    // and Tr[Gam G Gam G^H] = sum_jk (Gam G)_jk conj((G Gam)_jk) since Gam is Hermitian (FP64).
    cx<double>* D = reinterpret_cast<cx<double>*>(P->ws + P->L.dec);
    cx<double>* G64 = D;
    cx<double>* X1 = D + (size_t)P->Ec * bb;
    cx<double>* X2 = X1 + (size_t)P->Ec * bb;
    cx<double>* Dm = X2 + (size_t)P->Ec * bb;
    Term<T> tg; tg.p = c.g(0); tg.s = bb; tg.alpha = 1.0;
    QTX_CK((combine<T, double>(G64, bb, tg, none, none, b, ne, nullptr, 0, 0, nullptr, st)));
    Term<double> a0; a0.p = G64; a0.s = bb; a0.alpha = 1.0;
    Term<double> a1; a1.p = G64; a1.s = bb; a1.alpha = -1.0; a1.op = OP_C;
    Term<double> nn;
    QTX_CK((combine<double, double>(Dm, bb, a0, a1, nn, b, ne, nullptr, 0, 0, nullptr, st)));
    QTX_CK(obs_trace2<double>(tra, 1, Gam_L, bb, Dm, bb, nullptr, 0, nullptr, 0, b, ne, st, 1, -1.0));
    if ((s = gemm<double>(P, gargs<double>(b, b, b, Gam_L, b, bb, OP_N, G64, b, bb, OP_N, nullptr, 0, 0, X1, b, bb, 1.0, 0.0, ne, nullptr), st, true))) return s;
    if ((s = gemm<double>(P, gargs<double>(b, b, b, G64, b, bb, OP_N, Gam_L, b, bb, OP_N, nullptr, 0, 0, X2, b, bb, 1.0, 0.0, ne, nullptr), st, true))) return s;
    QTX_CK(obs_frob_dot(tra, 1, X1, bb, X2, bb, -1.0, b, ne, st));
  }
  return finish_chunk<T>(P, in, out, e0, ne, st);
}

template <typename T>
qtx_status solve_all(qtx_rgf_plan_s* P, const qtx_rgf_inputs* in, const qtx_rgf_outputs* out, cudaStream_t st) {
  const int nb = P->nb;
  const unsigned m = P->d.outputs;
  if ((m & QTX_OUT_INTEGRALS) && out->current_int && nb > 1)
    QTX_CK(cudaMemsetAsync(out->current_int, 0, (size_t)(nb - 1) * sizeof(double), st));
  if ((m & QTX_OUT_INTEGRALS) && out->density_int)
    QTX_CK(cudaMemsetAsync(out->density_int, 0, (size_t)nb * sizeof(double), st));
  int* chunk_status = reinterpret_cast<int*>(P->ws + P->L.flags) + 2 * P->Ec;
  P->status_host.assign(in->n_energies, 0);
  for (int e0 = 0; e0 < in->n_energies; e0 += P->Ec) {
    const int ne = std::min(P->Ec, in->n_energies - e0);
    int* status = out->status_per_energy ? out->status_per_energy + e0 : chunk_status;
    QTX_CK(cudaMemsetAsync(status, 0, (size_t)ne * sizeof(int), st));
    if (out->escalated) QTX_CK(cudaMemsetAsync(out->escalated + e0, 0, (size_t)ne * sizeof(int), st));
    qtx_status s = solve_chunk<T>(P, in, out, e0, ne, status, st);
    if (s) return s;
    if (!std::is_same<T, double>::value && P->d.escalate_tol > 0) {
      // energies whose current is not conserved to escalate_tol are solved again in FP64
      QTX_CK(cudaMemcpyAsync(P->h_flag, P->ws + P->L.cflag, sizeof(int) * ne, cudaMemcpyDeviceToHost, st));
      QTX_CK(cudaStreamSynchronize(st));
      std::vector<int> redo;
      for (int k = 0; k < ne; ++k)
        if (P->h_flag[k]) redo.push_back(k);
      if (!redo.empty()) {
        // take their integral contributions back out first (the chunk's per-energy values are still
        // in the observable buffers; each FP64 re-solve adds its own)
        const int nbm1 = nb - 1, ncur = nb > 1 ? nb - 1 : 1;
        double* cur = reinterpret_cast<double*>(P->ws + P->L.obs);
        double* den = cur + (size_t)P->Ec * ncur;
        if ((m & QTX_OUT_INTEGRALS) && out->current_int && nbm1 > 0)
          for (int k : redo)
            QTX_CK(integrate_add(out->current_int, cur + (size_t)k * ncur, ncur, nbm1, in->weights, in->energies, e0 + k,
                                 in->n_energies, 1, -1.0, st));
        if ((m & QTX_OUT_INTEGRALS) && out->density_int)
          for (int k : redo)
            QTX_CK(integrate_add(out->density_int, den + (size_t)k * nb, nb, nb, in->weights, in->energies, e0 + k,
                                 in->n_energies, 1, -1.0 / (2.0 * 3.14159265358979323846), st));
        for (int k : redo) {
          QTX_CK(cudaMemsetAsync(status + k, 0, sizeof(int), st));
          if ((s = solve_chunk<double>(P, in, out, e0 + k, 1, status + k, st))) return s;
          if (out->escalated) QTX_CK(fill_int(out->escalated + e0 + k, 1, 1, st));
        }
      }
    }
    if (!out->status_per_energy) {
      // keep the worst chunk status without a host sync: fold into the error flag word
      QTX_CK(cudaMemcpyAsync(P->h_status, status, sizeof(int) * ne, cudaMemcpyDeviceToHost, st));
      QTX_CK(cudaStreamSynchronize(st));
      for (int k = 0; k < ne; ++k) P->worst = std::max(P->worst, P->h_status[k]);
    }
  }
  return QTX_OK;
}

qtx_status validate(const qtx_rgf_desc* d, std::string& err) {
  if (!d) { err = "desc is NULL"; return QTX_ERR_INVALID_ARG; }
  if (d->n_blocks < 1) { err = "n_blocks must be >= 1"; return QTX_ERR_INVALID_ARG; }
  if (d->block_size < 1 || d->block_size > 4096) { err = "block_size must be in [1, 4096]"; return QTX_ERR_INVALID_ARG; }
  if (d->max_energies_in_flight < 1) { err = "max_energies_in_flight must be >= 1"; return QTX_ERR_INVALID_ARG; }
  if (d->precision < QTX_FP64 || d->precision > QTX_EMU64) { err = "unknown precision"; return QTX_ERR_INVALID_ARG; }
  if (d->leads && (d->decim_max_iter < 1 || !(d->decim_tol > 0))) { err = "leads need decim_max_iter >= 1 and decim_tol > 0"; return QTX_ERR_INVALID_ARG; }
  if (d->refine_max_iter < 0) { err = "refine_max_iter must be >= 0"; return QTX_ERR_INVALID_ARG; }
  if (!(d->refine_tol >= 0.0)) { err = "refine_tol must be >= 0"; return QTX_ERR_INVALID_ARG; }
  if (d->offdiag_sigma && !d->has_scattering) { err = "offdiag_sigma needs has_scattering"; return QTX_ERR_INVALID_ARG; }
  if (d->storage_bits && !fpx_width_ok(d->storage_bits)) { err = "storage_bits must be 0, 56, 48, 40, 32, 24 or 16"; return QTX_ERR_INVALID_ARG; }
  if (d->sigma_stream && (!d->has_scattering || !d->energy_dependent_sigma || d->offdiag_sigma)) { err = "sigma_stream needs has_scattering and energy_dependent_sigma, without offdiag_sigma"; return QTX_ERR_INVALID_ARG; }
  if (d->second_rhs && (!d->system_input || d->storage_bits)) { err = "second_rhs needs system_input and storage_bits = 0"; return QTX_ERR_INVALID_ARG; }
  if (!(d->escalate_tol >= 0.0)) { err = "escalate_tol must be >= 0"; return QTX_ERR_INVALID_ARG; }
  if (d->tc_stages < 0 || d->tc_ctas < 0) { err = "tc_stages and tc_ctas must be >= 0"; return QTX_ERR_INVALID_ARG; }
  if ((d->escalate_tol > 0 || (d->outputs & QTX_OUT_CONTINUITY)) && (d->offdiag_sigma || d->system_input || d->sigma_stream)) {
    err = "the continuity check (escalate_tol, QTX_OUT_CONTINUITY) needs block-diagonal Sigma, no system_input and no sigma_stream";
    return QTX_ERR_INVALID_ARG;
  }
  if (d->system_input) {
    const unsigned bad = (d->second_rhs ? 0u : QTX_OUT_GG_DIAG | QTX_OUT_GG_UPPER) | QTX_OUT_CURRENT | QTX_OUT_CONTACT | QTX_OUT_TRANSMISSION | QTX_OUT_INTEGRALS;
    if (d->has_S || d->leads || d->sigma_stream) { err = "system_input needs has_S = 0, leads = 0, sigma_stream = 0"; return QTX_ERR_INVALID_ARG; }
    if (d->outputs & bad) { err = "system_input produces no G^> (without second_rhs), current, contact, transmission or integrals outputs"; return QTX_ERR_INVALID_ARG; }
  }
  if ((d->precision == QTX_EMU64 || d->precision == QTX_BF16X3) && !tc_available()) {
    err = "tensor-core engine not compiled into the library";
    return QTX_ERR_UNSUPPORTED;
  }
  return QTX_OK;
}

}  // namespace

// ----------------------------------------------------------------------------- W-system assembly
// Table I, W row: per energy the BT blocks of M = I - V P^R and B^<> = V P^<> V^H from the exact
// block products of the BT factors.  Row i of V P is (V P)_ij = sum_k V_ik P_kj over k = i-1..i+1
// with |k - j| <= 1 (j = i-1..i+1 for M; i-2..i+2 for B, whose blocks B_ij = sum_l (V P)_il
// (V_jl)^H need l up to j+1).  Each block product is one batched launch over the chunk's energies,
// V shared (batch stride 0).  Temporaries: 0-4 V blocks, 5 one P block, 6-9 row i of V P, 10-11 B.
template <typename T>
qtx_status w_assemble_chunk(qtx_rgf_plan_s* P, const qtx_w_inputs* in, const qtx_w_outputs* out, int nb,
                            int e0, int ne, cudaStream_t st) {
  const int b = P->b;
  const long bb = P->bb, nu = nb - 1;
  Ctx<T> c{P, st, ne, nullptr, nullptr, bb, b};
  const cx<double>* Vd = reinterpret_cast<const cx<double>*>(in->V_diag);
  const cx<double>* Vu = reinterpret_cast<const cx<double>*>(in->V_upper);
  // block j of a per-energy array [N_E][n][b][b], first energy of the chunk
  auto pe = [&](const void* X, long n, long j) {
    return reinterpret_cast<const cx<double>*>(X) + ((long)e0 * n + j) * bb;
  };
  // V slots: 0 V_ii, 1 V_{i+1,i+1}, 2 V_{i-1,i}, 3 V_{i,i+1}, 4 V_{i+1,i+2}
  cx<T>* Vt[5] = {c.tmp(0), c.tmp(1), c.tmp(2), c.tmp(3), c.tmp(4)};
  cx<T>* Pt = c.tmp(5);
  cx<T>* acc[4] = {c.tmp(6), c.tmp(7), c.tmp(8), c.tmp(9)};  // (V P)_{i,i-1} .. (V P)_{i,i+2}
  cx<T>* Bt = c.tmp(11);
  cx<T>* Bu = c.tmp(10);
  auto toT = [&](cx<T>* dst, const cx<double>* src, long sSrc, int batch) {
    return axpby_from64<T>(dst, bb, src, sSrc, 1.0, nullptr, 0, 0.0, b, batch, st);
  };
  auto mm = [&](const cx<T>* A, long sA, int opA, const cx<T>* B, long sB, int opB, cx<T>* C, double al,
                bool first) {
    return gemm<T>(P, gargs<T>(b, b, b, A, b, sA, opA, B, b, sB, opB, first ? nullptr : C, b, bb, C, b, bb, al,
                               first ? 0.0 : 1.0, ne, nullptr), st);
  };
  // C (+)= al V_k op(P), P complex128 with batch stride sP: digitised as it is (df32 plans), or through Pt
  Prods<T> pr;
  auto addP = [&](const cx<T>* A, int opA, const cx<double>* Pb, long sP, int opB, cx<T>* C, double al, bool first) -> qtx_status {
    if constexpr (std::is_same<T, float>::value) {
      QTX_CK(toT(Pt, Pb, sP, ne));
      return mm(A, 0, opA, Pt, bb, opB, C, al, first);
    } else {
      GemmArgs<T> g = gargs<T>(b, b, b, A, b, 0, opA, reinterpret_cast<const cx<T>*>(Pb), b, sP, opB, first ? nullptr : C, b, bb, C,
                               b, bb, al, first ? 0.0 : 1.0, ne, nullptr);
      g.b64 = true;
      pr.add(g);
      return QTX_OK;
    }
  };
  // out[e][j] = alpha X (+ I), complex128, n blocks per energy
  auto emit64 = [&](void* dst, long n, long j, const cx<T>* X, double alpha, bool ident) -> qtx_status {
    cx<double>* o = reinterpret_cast<cx<double>*>(dst) + ((long)e0 * n + j) * bb;
    Term<T> t0; t0.p = X; t0.s = bb; t0.alpha = alpha;
    Term<T> none;
    QTX_CK((combine<T, double>(o, n * bb, t0, none, none, b, ne, nullptr, 0.0, 0.0, nullptr, st)));
    if (ident) QTX_CK(add_identity<double>(o, n * bb, b, ne, nullptr, st));
    return QTX_OK;
  };
  qtx_status s;
  for (int i = 0; i < nb; ++i) {
    QTX_CK(toT(Vt[0], Vd + (long)i * bb, 0, 1));
    if (i + 1 < nb) QTX_CK(toT(Vt[1], Vd + (long)(i + 1) * bb, 0, 1));
    if (i >= 1) QTX_CK(toT(Vt[2], Vu + (long)(i - 1) * bb, 0, 1));
    if (i + 1 < nb) QTX_CK(toT(Vt[3], Vu + (long)i * bb, 0, 1));
    if (i + 2 < nb) QTX_CK(toT(Vt[4], Vu + (long)(i + 1) * bb, 0, 1));
    // row i of V P for j = i+j0 .. i+j1.  V_ik: k = i-1 -> V_{i-1,i}^H, k = i -> V_ii, k = i+1 -> V_{i,i+1}.
    // P_kj: diagonal, upper (j = k+1), lower (j = k-1): given, or -(P_{j,j+1})^H for anti-Hermitian P.
    // The sums over k of different j are independent: their n-th terms are launched together.
    auto row = [&](const void* Pd, const void* Pu, const void* Pl, int j0, int j1) -> qtx_status {
      for (int term = 0; term < 3; ++term) {
        for (int j = std::max(i + j0, 0); j <= std::min(i + j1, nb - 1); ++j) {
          const int k = std::max({i - 1, j - 1, 0}) + term;  // k in [i-1, i+1] and [j-1, j+1]
          if (k > std::min({i + 1, j + 1, nb - 1})) continue;
          const cx<T>* Vk = k == i ? Vt[0] : (k == i + 1 ? Vt[3] : Vt[2]);
          const int opV = k == i - 1 ? OP_C : OP_N;
          cx<T>* C = acc[j - i + 1];
          if (k == j) s = addP(Vk, opV, pe(Pd, nb, k), (long)nb * bb, OP_N, C, 1.0, term == 0);
          else if (j == k + 1) s = addP(Vk, opV, pe(Pu, nu, k), nu * bb, OP_N, C, 1.0, term == 0);
          else if (Pl) s = addP(Vk, opV, pe(Pl, nu, j), nu * bb, OP_N, C, 1.0, term == 0);
          else s = addP(Vk, opV, pe(Pu, nu, j), nu * bb, OP_C, C, -1.0, term == 0);
          if (s) return s;
        }
        if ((s = run<T>(P, pr, st))) return s;
      }
      return QTX_OK;
    };
    // M_ii = I - (V P^R)_ii, M_{i,i+1} = -(V P^R)_{i,i+1}, M_{i,i-1} = -(V P^R)_{i,i-1}
    if ((s = row(in->PR_diag, in->PR_upper, in->PR_lower, -1, 1))) return s;
    if ((s = emit64(out->M_diag, nb, i, acc[1], -1.0, true))) return s;
    if (i + 1 < nb && (s = emit64(out->M_upper, nu, i, acc[2], -1.0, false))) return s;
    if (i >= 1 && (s = emit64(out->M_lower, nu, i - 1, acc[0], -1.0, false))) return s;
    for (int kind = 0; kind < 2; ++kind) {
      const void* Pd = kind ? in->PG_diag : in->PL_diag;
      const void* Pu = kind ? in->PG_upper : in->PL_upper;
      void* Od = kind ? out->BG_diag : out->BL_diag;
      void* Ou = kind ? out->BG_upper : out->BL_upper;
      if (!Pd) continue;
      if ((s = row(Pd, Pu, nullptr, -1, 2))) return s;  // B's blocks need (V P)_il for l = i-1 .. i+2
      // B_ii = sum_l (V P)_il (V_il)^H, l = i-1..i+1:  (V_{i,i-1})^H = V_{i-1,i}, V_ii^H, V_{i,i+1}^H
      // B_{i,i+1} = sum_l (V P)_il (V_{i+1,l})^H, l = i..i+2:  V_{i,i+1}, V_{i+1,i+1}^H, V_{i+1,i+2}^H
      // (the two sums' n-th terms together)
      auto close = [&](int l, const cx<T>* Vl, int op, cx<T>* C, bool first) {
        pr.add(gargs<T>(b, b, b, acc[l - i + 1], b, bb, OP_N, Vl, b, 0, op, first ? nullptr : C, b, bb, C, b, bb, 1.0,
                        first ? 0.0 : 1.0, ne, nullptr));
      };
      const int d0 = std::max(i - 1, 0);
      for (int term = 0; term < 3; ++term) {
        const int ld = d0 + term, lu = i + term;
        if (ld <= std::min(i + 1, nb - 1))
          close(ld, ld == i ? Vt[0] : (ld == i + 1 ? Vt[3] : Vt[2]), ld == i - 1 ? OP_N : OP_C, Bt, term == 0);
        if (i + 1 < nb && lu <= std::min(i + 2, nb - 1))
          close(lu, lu == i ? Vt[3] : (lu == i + 1 ? Vt[1] : Vt[4]), lu == i ? OP_N : OP_C, Bu, term == 0);
        if ((s = run<T>(P, pr, st))) return s;
      }
      if ((s = emit64(Od, nb, i, Bt, 1.0, false))) return s;
      if (i + 1 < nb && (s = emit64(Ou, nu, i, Bu, 1.0, false))) return s;
    }
  }
  return QTX_OK;
}

extern "C" {

qtx_status qtx_rgf_plan_create(const qtx_rgf_desc* desc, qtx_rgf_plan* out) {
  if (!out) { g_create_error = "out is NULL"; return QTX_ERR_INVALID_ARG; }
  *out = nullptr;
  std::string err;
  qtx_status s = validate(desc, err);
  if (s) { g_create_error = err; return s; }
  auto* P = new qtx_rgf_plan_s();
  P->d = *desc;
  P->b = desc->block_size;
  P->nb = desc->n_blocks;
  P->Ec = desc->max_energies_in_flight;
  P->bb = (long)P->b * P->b;
  P->esz = desc->precision == QTX_FP32 ? sizeof(cx<float>) : sizeof(cx<double>);
  P->L = make_layout(*desc);
  cudaError_t e = cudaMalloc(&P->ws, P->L.total);
  if (e != cudaSuccess) {
    g_create_error = std::string("workspace cudaMalloc(") + std::to_string(P->L.total) + "): " + cudaGetErrorString(e);
    cudaGetLastError();
    delete P;
    return QTX_ERR_OOM;
  }
  e = cudaMalloc(&P->d_err_flag, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(P->d_err_flag, 0, sizeof(int));
  if (e == cudaSuccess) e = cudaMallocHost(&P->h_status, sizeof(int) * P->Ec);
  if (e == cudaSuccess && desc->escalate_tol > 0) e = cudaMallocHost(&P->h_flag, sizeof(int) * P->Ec);
  // identity block for the refinement residual (plans whose inverses are refined)
  if (e == cudaSuccess && P->L.refine64)
    e = set_identity(reinterpret_cast<cx<double>*>(P->ws + P->L.ident), reinterpret_cast<cx<df>*>(P->ws + P->L.ident_df), P->b, nullptr);
  if (e == cudaSuccess && P->L.refine64) e = cudaStreamSynchronize(nullptr);
  if (e != cudaSuccess) {
    g_create_error = std::string("plan setup: ") + cudaGetErrorString(e);
    cudaFree(P->ws);
    if (P->d_err_flag) cudaFree(P->d_err_flag);
    if (P->h_status) cudaFreeHost(P->h_status);
    if (P->h_flag) cudaFreeHost(P->h_flag);
    delete P;
    return QTX_ERR_CUDA;
  }
  *out = P;
  return QTX_OK;
}

qtx_status qtx_rgf_solve(qtx_rgf_plan P, const qtx_rgf_inputs* in, const qtx_rgf_outputs* out, void* stream) {
  if (!P) return QTX_ERR_INVALID_ARG;
  if (!in || !out) { P->err = "inputs/outputs NULL"; return QTX_ERR_INVALID_ARG; }
  if (in->n_energies < 1 || !in->energies) { P->err = "need n_energies >= 1 and an energies array"; return QTX_ERR_INVALID_ARG; }
  const int nbs = in->n_blocks ? in->n_blocks : P->d.n_blocks;
  if (P->d.system_input) {
    if (!in->M_diag || (nbs > 1 && (!in->M_upper || !in->M_lower))) { P->err = "system_input set but M blocks missing"; return QTX_ERR_INVALID_ARG; }
  } else if (!in->H_diag || (nbs > 1 && !in->H_upper)) { P->err = "H_diag / H_upper missing"; return QTX_ERR_INVALID_ARG; }
  if (P->d.has_S && (!in->S_diag || (P->nb > 1 && !in->S_upper))) { P->err = "has_S set but S pointers missing"; return QTX_ERR_INVALID_ARG; }
  if (P->d.has_scattering && (!in->SigL_diag || (!P->d.system_input && !in->SigR_diag))) { P->err = "has_scattering set but Sigma pointers missing"; return QTX_ERR_INVALID_ARG; }
  if (P->d.offdiag_sigma && (in->n_blocks ? in->n_blocks : P->d.n_blocks) > 1 &&
      (!in->SigL_upper || (!P->d.system_input && (!in->SigR_upper || !in->SigR_lower)))) { P->err = "offdiag_sigma set but off-diagonal Sigma pointers missing"; return QTX_ERR_INVALID_ARG; }
  if (P->d.second_rhs && (!in->SigG_diag || (P->d.offdiag_sigma && nbs > 1 && !in->SigG_upper))) { P->err = "second_rhs set but SigG blocks missing"; return QTX_ERR_INVALID_ARG; }
  if (P->d.leads && (!in->lead_H00_L || !in->lead_H01_L || !in->lead_H00_R || !in->lead_H01_R)) { P->err = "leads set but lead blocks missing"; return QTX_ERR_INVALID_ARG; }
  if (P->d.leads && !(in->kT > 0)) { P->err = "leads need kT > 0"; return QTX_ERR_INVALID_ARG; }
  if (in->n_blocks < 0 || in->n_blocks > P->d.n_blocks) { P->err = "inputs->n_blocks exceeds the plan's n_blocks"; return QTX_ERR_INVALID_ARG; }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  P->last = st;
  P->worst = 0;
  EarlyLaunches early(P->L.short_launches && !P->group ? 2 : 1);
  // the bounded-wait flag of the tensor-core launches starts clear for every solve
  if (cudaMemsetAsync(P->d_err_flag, 0, sizeof(int), st) != cudaSuccess) {
    P->err = "clearing the wait flag failed";
    cudaGetLastError();
    return QTX_ERR_CUDA;
  }
  // the workspace is laid out for the plan's n_blocks; a shorter device uses its first slices
  P->nb = in->n_blocks ? in->n_blocks : P->d.n_blocks;
  qtx_status s;
  if (P->d.precision == QTX_FP32) s = solve_all<float>(P, in, out, st);
  else if (P->d.precision == QTX_FP64) s = solve_all<double>(P, in, out, st);
  else s = solve_all<df>(P, in, out, st);
  P->nb = P->d.n_blocks;
  if (s == QTX_OK) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { P->err = cudaGetErrorString(e); return QTX_ERR_CUDA; }
  }
  P->out_status = out->status_per_energy;
  P->out_status_n = in->n_energies;
  return s;
}

qtx_status qtx_w_assemble(qtx_rgf_plan P, const qtx_w_inputs* in, const qtx_w_outputs* out, void* stream) {
  if (!P) return QTX_ERR_INVALID_ARG;
  if (!in || !out) { P->err = "inputs/outputs NULL"; return QTX_ERR_INVALID_ARG; }
  const int nb = in->n_blocks ? in->n_blocks : P->d.n_blocks;
  if (in->n_blocks < 0 || nb > P->d.n_blocks || in->n_energies < 1) { P->err = "n_blocks / n_energies out of range"; return QTX_ERR_INVALID_ARG; }
  if (!in->V_diag || !in->PR_diag || !in->PL_diag || !out->M_diag || !out->BL_diag) { P->err = "W assembly: diagonal blocks missing"; return QTX_ERR_INVALID_ARG; }
  if (nb > 1 && (!in->V_upper || !in->PR_upper || !in->PR_lower || !in->PL_upper || !out->M_upper || !out->M_lower || !out->BL_upper)) {
    P->err = "W assembly: off-diagonal blocks missing";
    return QTX_ERR_INVALID_ARG;
  }
  const bool pg = in->PG_diag != nullptr;
  if ((!pg && in->PG_upper) || (pg && ((nb > 1 && !in->PG_upper) || !out->BG_diag || (nb > 1 && !out->BG_upper)))) {
    P->err = "W assembly: P^> (diagonal and upper) and B^> must come together";
    return QTX_ERR_INVALID_ARG;
  }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  P->last = st;
  EarlyLaunches early(P->L.short_launches && !P->group ? 2 : 1);
  if (cudaMemsetAsync(P->d_err_flag, 0, sizeof(int), st) != cudaSuccess) {
    P->err = "clearing the wait flag failed";
    cudaGetLastError();
    return QTX_ERR_CUDA;
  }
  for (int e0 = 0; e0 < in->n_energies; e0 += P->Ec) {
    const int ne = std::min(P->Ec, in->n_energies - e0);
    qtx_status s;
    if (P->d.precision == QTX_FP32) s = w_assemble_chunk<float>(P, in, out, nb, e0, ne, st);
    else if (P->d.precision == QTX_FP64) s = w_assemble_chunk<double>(P, in, out, nb, e0, ne, st);
    else s = w_assemble_chunk<df>(P, in, out, nb, e0, ne, st);
    if (s) return s;
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { P->err = cudaGetErrorString(e); return QTX_ERR_CUDA; }
  return QTX_OK;
}

qtx_status qtx_rgf_status(qtx_rgf_plan P) {
  if (!P) return QTX_ERR_INVALID_ARG;
  cudaError_t e = cudaStreamSynchronize(P->last);
  if (e != cudaSuccess) { P->err = cudaGetErrorString(e); return QTX_ERR_CUDA; }
  int flag = 0;
  e = cudaMemcpy(&flag, P->d_err_flag, sizeof(int), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) { P->err = cudaGetErrorString(e); return QTX_ERR_CUDA; }
  if (flag) { P->err = "tensor-core engine: bounded wait expired"; return QTX_ERR_TIMEOUT; }
  if (P->out_status) {
    P->status_host.assign(P->out_status_n, 0);
    e = cudaMemcpy(P->status_host.data(), P->out_status, sizeof(int) * P->out_status_n, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) { P->err = cudaGetErrorString(e); return QTX_ERR_CUDA; }
    for (int v : P->status_host) P->worst = std::max(P->worst, v);
  }
  return (qtx_status)P->worst;
}

qtx_status qtx_rgf_set_profiling(qtx_rgf_plan P, int enable) {
  if (!P) return QTX_ERR_INVALID_ARG;
  P->prof = enable != 0;
  P->ev_used = 0;
  P->pipe_flops = P->useful_flops = 0.0;
  return QTX_OK;
}

qtx_status qtx_rgf_gemm_profile(qtx_rgf_plan P, long long* launches, double* ms, double* pipe_flops,
                                double* useful_flops) {
  if (!P) return QTX_ERR_INVALID_ARG;
  double tot = 0.0;
  for (size_t k = 0; k + 1 < P->ev_used; k += 2) {
    cudaError_t e = cudaEventSynchronize(P->ev_pool[k + 1]);
    float t = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&t, P->ev_pool[k], P->ev_pool[k + 1]);
    if (e != cudaSuccess) { P->err = cudaGetErrorString(e); return QTX_ERR_CUDA; }
    tot += t;
  }
  if (launches) *launches = (long long)(P->ev_used / 2);
  if (ms) *ms = tot;
  if (pipe_flops) *pipe_flops = P->pipe_flops;
  if (useful_flops) *useful_flops = P->useful_flops;
  P->ev_used = 0;
  P->pipe_flops = P->useful_flops = 0.0;
  return QTX_OK;
}

long long qtx_kernel_launches(void) { return g_launches.load(); }

qtx_status qtx_rgf_destroy(qtx_rgf_plan P) {
  if (!P) return QTX_OK;
  for (cudaEvent_t e : P->ev_pool) cudaEventDestroy(e);
  if (P->ws) cudaFree(P->ws);
  if (P->d_err_flag) cudaFree(P->d_err_flag);
  if (P->h_status) cudaFreeHost(P->h_status);
  if (P->h_flag) cudaFreeHost(P->h_flag);
  delete P;
  return QTX_OK;
}

const char* qtx_rgf_last_error(qtx_rgf_plan P) { return P ? P->err.c_str() : g_create_error.c_str(); }

size_t qtx_rgf_footprint(const qtx_rgf_desc* desc) {
  std::string err;
  if (validate(desc, err) && validate(desc, err) != QTX_ERR_UNSUPPORTED) return 0;
  return make_layout(*desc).total;
}

const char* qtx_rgf_version(void) { return "qtx-rgf 0.1 (sm_103a)"; }

}  // extern "C"

// ============================================================================ component ABI
namespace {

// Temporaries of the component calls come from a memory pool of the library's own (one per device): the
// default pool returns everything to the driver at each synchronisation, and these calls synchronise, so
// every call paid for mapping its memory again (0.9 ms of a 1.2 ms product).  The pool keeps at most kPoolKeep
// between calls and gives the rest back; allocation and reuse are stream-ordered, so calls on several
// streams and threads share it.  qtx_release_memory gives the rest back too, and CUDA takes it for an allocation of this
// process that would not fit beside it.
constexpr unsigned long long kPoolKeep = 512ull << 20;
// make = false: the pool of the current device and context if there is one, else an error
cudaError_t component_pool(cudaMemPool_t* out, bool make = true) {
  struct Entry {
    int dev;
    unsigned long long ctx;  // ids are not used again: one of a context that cudaDeviceReset ended matches no other
    cudaMemPool_t pool;
  };
  static std::mutex mu;
  static std::vector<Entry> pools;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(mu);
  const unsigned long long ctx = current_ctx_id();
  for (const Entry& p : pools)
    if (p.dev == dev && p.ctx == ctx) {
      *out = p.pool;
      return cudaSuccess;
    }
  if (!make) return cudaErrorInvalidValue;
  cudaMemPoolProps props = {};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaMemPool_t p;
  if ((e = cudaMemPoolCreate(&p, &props)) != cudaSuccess) return e;
  unsigned long long keep = kPoolKeep;
  if ((e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep)) != cudaSuccess) {
    cudaMemPoolDestroy(p);
    return e;
  }
  pools.push_back({dev, current_ctx_id(), p});  // (the pool's creation made a context if there was none)
  *out = p;
  return cudaSuccess;
}
// Stream-ordered temporaries of one call, freed when it returns.
struct Temps {
  cudaStream_t st;
  cudaMemPool_t pool = nullptr;
  cudaError_t e;
  std::vector<void*> held;
  explicit Temps(cudaStream_t s) : st(s), e(component_pool(&pool)) {}
  template <typename T>
  T* get(size_t count) {
    void* p = nullptr;
    if (e == cudaSuccess && count) e = cudaMallocFromPoolAsync(&p, count * sizeof(T), pool, st);
    if (p) held.push_back(p);
    return static_cast<T*>(p);
  }
  ~Temps() {
    for (void* p : held) cudaFreeAsync(p, st);
  }
};

// whether two batched arrays of complex128 matrices share addresses
struct Span {
  uintptr_t lo, hi;
  Span(const void* p, int rows, int cols, long ld, long s, int n) {
    const long row = (long)(rows - 1) * ld, ent = (long)(n - 1) * s;
    lo = (uintptr_t)((const cx<double>*)p + std::min(0L, row) + std::min(0L, ent));
    hi = (uintptr_t)((const cx<double>*)p + std::max(0L, row) + std::max(0L, ent) + cols);
  }
  bool meets(const Span& o) const { return lo < o.hi && o.lo < hi; }
};

// FP64, EMU64 and BF16X3 products: straight from the caller's complex128 arrays, straight into C unless C
// shares addresses with an operand (or with C0 in another layout), which then goes through a copy.
qtx_status zgemm_direct(int precision, GemmArgs<double> g, cudaStream_t st, std::string& err) {
  const bool emu = precision != QTX_FP64;
  const bool tc = emu || (g.M >= kTcF64Min && g.N >= kTcF64Min && g.K >= kTcF64Min && tc_available());
  const int rA = g.opA == OP_N ? g.M : g.K, cA = g.opA == OP_N ? g.K : g.M;
  const int rB = g.opB == OP_N ? g.K : g.N, cB = g.opB == OP_N ? g.N : g.K;
  const Span sc(g.C, g.M, g.N, g.ldc, g.sC, g.batch);
  bool clash = g.K > 0 && (sc.meets(Span(g.A, rA, cA, g.lda, g.sA, g.sA ? g.batch : 1)) ||
                           sc.meets(Span(g.B, rB, cB, g.ldb, g.sB, g.sB ? g.batch : 1)));
  if (g.C0 && !(g.C0 == g.C && g.ldc0 == g.ldc && g.sC0 == g.sC))
    clash |= sc.meets(Span(g.C0, g.M, g.N, g.ldc0, g.sC0, g.sC0 ? g.batch : 1));
  const int digits = precision == QTX_EMU64 ? 6 : 2;
  const size_t bytes = !tc ? 0 : (emu ? gemm_tc_scratch_bytes(g.M, g.N, g.K, g.batch, digits)
                                      : gemm_fp64_tc_scratch_bytes(g.M, g.N, g.K, g.batch));
  Temps t(st);
  unsigned char* scr = t.get<unsigned char>(bytes);
  int* flag = t.get<int>(1);
  cx<double>* C = clash ? t.get<cx<double>>((size_t)g.batch * g.M * g.N) : g.C;
  cudaError_t e = t.e;
  GemmArgs<double> w = g;
  if (clash) {
    w.C = C;
    w.ldc = g.N;
    w.sC = (long)g.M * g.N;
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(flag, 0, sizeof(int), st);
  if (e == cudaSuccess) {
    if (emu) {
      TcArgs a;
      a.M = w.M; a.N = w.N; a.K = w.K;
      a.ta = a.tb = a.tc = EL_F64;
      a.A = reinterpret_cast<const cx<df>*>(w.A); a.lda = w.lda; a.sA = w.sA; a.opA = w.opA;
      a.B = reinterpret_cast<const cx<df>*>(w.B); a.ldb = w.ldb; a.sB = w.sB; a.opB = w.opB;
      a.C0 = reinterpret_cast<const cx<df>*>(w.C0); a.ldc0 = w.ldc0; a.sC0 = w.sC0;
      a.C = reinterpret_cast<cx<df>*>(w.C); a.ldc = w.ldc; a.sC = w.sC;
      a.alpha = w.alpha; a.beta = w.beta;
      a.batch = w.batch; a.active = nullptr;
      e = gemm_tc(a, digits, scr, bytes, flag, st);
    } else {
      e = tc ? gemm_fp64_tc(w, scr, bytes, flag, st) : gemm_simt<double>(w, st);
    }
  }
  if (e == cudaSuccess && clash)
    e = convert_strided<double, double>(C, g.N, (long)g.M * g.N, g.C, g.ldc, g.sC, g.M, g.N, g.batch, st);
  int hflag = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&hflag, flag, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    err = cudaGetErrorString(e);
    cudaGetLastError();
    return QTX_ERR_CUDA;
  }
  if (hflag) { err = "tensor-core engine: bounded wait expired"; return QTX_ERR_TIMEOUT; }
  return QTX_OK;
}

// FP32 products: operands rounded to complex64 copies, the result widened into C.
qtx_status zgemm_f32(const GemmArgs<double>& g, cudaStream_t st, std::string& err) {
  const int rA = g.opA == OP_N ? g.M : g.K, cA = g.opA == OP_N ? g.K : g.M;
  const int rB = g.opB == OP_N ? g.K : g.N, cB = g.opB == OP_N ? g.N : g.K;
  const int nA = g.sA ? g.batch : 1, nB = g.sB ? g.batch : 1, nC0 = g.C0 ? (g.sC0 ? g.batch : 1) : 0;
  Temps t(st);
  cx<float>* a = t.get<cx<float>>((size_t)nA * rA * cA);
  cx<float>* b = t.get<cx<float>>((size_t)nB * rB * cB);
  cx<float>* c0 = t.get<cx<float>>((size_t)nC0 * g.M * g.N);
  cx<float>* c = t.get<cx<float>>((size_t)g.batch * g.M * g.N);
  cudaError_t e = t.e;
  if (e == cudaSuccess) e = convert_strided<double, float>(g.A, g.lda, g.sA, a, cA, (long)rA * cA, rA, cA, nA, st);
  if (e == cudaSuccess) e = convert_strided<double, float>(g.B, g.ldb, g.sB, b, cB, (long)rB * cB, rB, cB, nB, st);
  if (e == cudaSuccess && nC0) e = convert_strided<double, float>(g.C0, g.ldc0, g.sC0, c0, g.N, (long)g.M * g.N, g.M, g.N, nC0, st);
  if (e == cudaSuccess)
    e = gemm_simt<float>(gargs<float>(g.M, g.N, g.K, a, cA, nA > 1 ? (long)rA * cA : 0, g.opA, b, cB, nB > 1 ? (long)rB * cB : 0,
                                      g.opB, nC0 ? c0 : nullptr, g.N, nC0 > 1 ? (long)g.M * g.N : 0, c, g.N, (long)g.M * g.N,
                                      g.alpha, g.beta, g.batch, nullptr), st);
  if (e == cudaSuccess) e = convert_strided<float, double>(c, g.N, (long)g.M * g.N, g.C, g.ldc, g.sC, g.M, g.N, g.batch, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    err = cudaGetErrorString(e);
    cudaGetLastError();
    return QTX_ERR_CUDA;
  }
  return QTX_OK;
}

template <typename T>
qtx_status zinv_via(qtx_rgf_plan_s* P, int n, void* A, long sA, int batch, int* status, cudaStream_t st) {
  cx<T>* X = reinterpret_cast<cx<T>*>(P->ws + P->L.g);
  const long nn = (long)n * n;
  QTX_CK((convert_strided<double, T>((const cx<double>*)A, n, sA, X, n, nn, n, n, batch, st)));
  qtx_status s = block_inverse<T>(P, X, n, batch, nullptr, status, st);
  if (s) return s;
  QTX_CK((convert_strided<T, double>(X, n, nn, (cx<double>*)A, n, sA, n, n, batch, st)));
  return QTX_OK;
}
template <>
qtx_status zinv_via<double>(qtx_rgf_plan_s* P, int n, void* A, long sA, int batch, int* status, cudaStream_t st) {
  cx<double>* X = reinterpret_cast<cx<double>*>(P->ws + P->L.g);
  const long nn = (long)n * n;
  QTX_CK(cudaMemcpy2DAsync(X, nn * sizeof(cx<double>), A, sA * sizeof(cx<double>), nn * sizeof(cx<double>), batch,
                           cudaMemcpyDeviceToDevice, st));
  qtx_status s = block_inverse<double>(P, X, n, batch, nullptr, status, st);
  if (s) return s;
  QTX_CK(cudaMemcpy2DAsync(A, sA * sizeof(cx<double>), X, nn * sizeof(cx<double>), nn * sizeof(cx<double>), batch,
                           cudaMemcpyDeviceToDevice, st));
  return QTX_OK;
}

thread_local std::string g_kernel_error;

}  // namespace

extern "C" {

qtx_status qtx_zgemm_batched(int precision, int M, int N, int K, int opA, const void* A, long lda, long sA, int opB,
                             const void* B, long ldb, long sB, double alpha, double beta, const void* C0, long ldc0,
                             long sC0, void* C, long ldc, long sC, int batch, void* stream) {
  if (M < 0 || N < 0 || K < 0 || batch < 1 || !A || !B || !C || (beta != 0.0 && !C0) ||
      (opA != OP_N && opA != OP_C) || (opB != OP_N && opB != OP_C)) {
    g_kernel_error = "qtx_zgemm_batched: invalid argument";
    return QTX_ERR_INVALID_ARG;
  }
  if (M == 0 || N == 0) return QTX_OK;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const bool c0 = C0 && beta != 0.0;
  const GemmArgs<double> g = gargs<double>(M, N, K, (const cx<double>*)A, lda, sA, opA, (const cx<double>*)B, ldb, sB, opB,
                                           c0 ? (const cx<double>*)C0 : nullptr, ldc0, sC0, (cx<double>*)C, ldc, sC, alpha,
                                           c0 ? beta : 0.0, batch, nullptr);
  switch (precision) {
    case QTX_FP32: return zgemm_f32(g, st, g_kernel_error);
    case QTX_EMU64:
    case QTX_BF16X3:
      if (!tc_available()) { g_kernel_error = "tensor-core engine needs an sm_103 GPU"; return QTX_ERR_UNSUPPORTED; }
      return zgemm_direct(precision, g, st, g_kernel_error);
    case QTX_FP64: return zgemm_direct(precision, g, st, g_kernel_error);
    default:
      g_kernel_error = "unknown precision";
      return QTX_ERR_INVALID_ARG;
  }
}

qtx_status qtx_release_memory(void) {
  cudaMemPool_t p = nullptr;
  if (component_pool(&p, false) != cudaSuccess) return QTX_OK;  // none yet
  // (a block counts as free once the host has seen its free complete)
  if (cudaDeviceSynchronize() == cudaSuccess && cudaMemPoolTrimTo(p, 0) == cudaSuccess) return QTX_OK;
  cudaGetLastError();
  return QTX_ERR_CUDA;
}

qtx_status qtx_zinv_batched(int precision, int n, void* A, long sA, int batch, int refine_iter, int* status, void* stream) {
  if (n < 1 || n > 4096 || batch < 1 || !A || refine_iter < 0) return QTX_ERR_INVALID_ARG;
  qtx_rgf_desc d{};
  d.n_blocks = 1;
  d.block_size = n;
  d.max_energies_in_flight = batch;
  d.precision = (qtx_precision)precision;
  d.refine_max_iter = refine_iter;
  std::string err;
  qtx_status s = validate(&d, err);
  if (s) { g_create_error = err; return s; }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  // a plan of the inverse's areas alone, in stream-ordered memory
  qtx_rgf_plan_s plan;
  qtx_rgf_plan_s* P = &plan;
  P->d = d;
  P->b = n;
  P->nb = 1;
  P->Ec = batch;
  P->bb = (long)n * n;
  P->esz = precision == QTX_FP32 ? sizeof(cx<float>) : sizeof(cx<double>);
  P->L = make_layout(d, true);
  Temps t(st);
  P->ws = t.get<unsigned char>(P->L.total);
  P->d_err_flag = t.get<int>(1);
  if (t.e != cudaSuccess) {
    g_create_error = std::string("workspace of ") + std::to_string(P->L.total) + " bytes: " + cudaGetErrorString(t.e);
    cudaGetLastError();
    return QTX_ERR_OOM;
  }
  cudaError_t e = cudaMemsetAsync(P->d_err_flag, 0, sizeof(int), st);
  if (e == cudaSuccess && P->L.refine64)
    e = set_identity(reinterpret_cast<cx<double>*>(P->ws + P->L.ident), reinterpret_cast<cx<df>*>(P->ws + P->L.ident_df), n, st);
  int* stat = status;
  if (!stat) stat = reinterpret_cast<int*>(P->ws + P->L.flags);
  if (e == cudaSuccess && !status) e = cudaMemsetAsync(stat, 0, sizeof(int) * batch, st);
  if (e != cudaSuccess) { cudaGetLastError(); return QTX_ERR_CUDA; }
  if (precision == QTX_FP32) s = zinv_via<float>(P, n, A, sA, batch, stat, st);
  else if (precision == QTX_FP64) s = zinv_via<double>(P, n, A, sA, batch, stat, st);
  else s = zinv_via<df>(P, n, A, sA, batch, stat, st);
  int hflag = 0;  // raised by a tensor-core product whose bounded wait expired
  if (s == QTX_OK && P->L.tc_bytes && cudaMemcpyAsync(&hflag, P->d_err_flag, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) s = QTX_ERR_CUDA;
  e = cudaStreamSynchronize(st);
  if (s == QTX_OK && e != cudaSuccess) s = QTX_ERR_CUDA;
  if (s == QTX_OK && hflag) {
    g_create_error = "tensor-core engine: bounded wait expired";
    s = QTX_ERR_TIMEOUT;
  }
  return s;
}

qtx_status qtx_lead_self_energy(int n, const void* H00, const void* H01, const double* energies, int n_energies,
                                double eta, double tol, int max_iter, void* SigR, int* status, void* stream) {
  if (n < 1 || n > 4096 || n_energies < 1 || !H00 || !H01 || !energies || !SigR || max_iter < 1 || !(tol > 0))
    return QTX_ERR_INVALID_ARG;
  qtx_rgf_desc d{};
  d.n_blocks = 1;
  d.block_size = n;
  d.max_energies_in_flight = n_energies;
  d.precision = QTX_FP64;
  d.leads = 1;
  d.decim_tol = tol;
  d.decim_max_iter = max_iter;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  std::string err;
  qtx_status s = validate(&d, err);
  if (s) { g_create_error = err; return s; }
  qtx_rgf_plan_s plan;  // the contact's and the inverse's areas alone, in stream-ordered memory
  qtx_rgf_plan_s* P = &plan;
  P->d = d;
  P->b = n;
  P->nb = 1;
  P->Ec = n_energies;
  P->bb = (long)n * n;
  P->esz = sizeof(cx<double>);
  P->L = make_layout(d, true);
  Temps t(st);
  P->ws = t.get<unsigned char>(P->L.total);
  P->d_err_flag = t.get<int>(1);
  if (t.e != cudaSuccess) {
    g_create_error = std::string("workspace of ") + std::to_string(P->L.total) + " bytes: " + cudaGetErrorString(t.e);
    cudaGetLastError();
    return QTX_ERR_OOM;
  }
  int* stat = status ? status : reinterpret_cast<int*>(P->ws + P->L.flags) + 2 * P->Ec;
  cudaMemsetAsync(stat, 0, sizeof(int) * n_energies, st);
  Ctx<double> c{P, st, n_energies, energies, stat, (long)n * n, n};
  const cx<double>*h00 = (const cx<double>*)H00, *h01 = (const cx<double>*)H01;
  cx<double>* sr = (cx<double>*)SigR;
  s = contacts<double>(c, 1, &h00, &h01, eta, &sr);
  cudaError_t e = cudaStreamSynchronize(st);
  if (s == QTX_OK && e != cudaSuccess) s = QTX_ERR_CUDA;
  return s;
}

}  // extern "C"

// ----------------------------------------------------------------------------- groups (uneven batches)
// Several plans -- devices of different N_B and b, each with its own energies -- solved together:
// every member's solve runs on its own host thread and stream, so the streams' launches overlap on
// the GPU.  With a pooling threshold of w > 0 waves, a tensor-core product is digitised on the
// member's stream; if it fills at least w waves of the GPU alone it is launched there at once,
// otherwise it is pooled: the member posts it and waits, and the pending products are launched
// together -- one persistent kernel over the union of their tiles, per kernel variant, at most
// kTcMaxGroup products a launch -- on the group's stream once they fill w waves, once every member
// still solving has posted one, or once the poster has waited kPoolWaitUs on the host.  Events order
// each pooled launch after its members' preceding work and before their following work.  The
// grouping only changes which launch computes a tile, never how, so every member's results equal
// its plan's solo solve bit for bit; the launches are plain stream work joined back to the caller's
// stream, so a group solve can be captured in a CUDA graph.  Pooling is off by default: its events
// hold the members in step, which costs more than the merged launches save.
constexpr int kPoolWaves = 0;  // default pooling threshold (qtx_rgf_group_set_pool_waves)
constexpr int kPoolWaitUs = 50;

struct qtx_rgf_group_s {
  std::vector<qtx_rgf_plan_s*> plans;
  std::vector<cudaStream_t> mst;     // member streams
  std::vector<cudaEvent_t> ready;    // per member: its work up to the posted product
  cudaStream_t gst = nullptr;        // launch stream of the pooled products
  std::vector<cudaEvent_t> done;     // ring of launch events
  size_t done_pos = 0;
  cudaEvent_t fork = nullptr;
  std::vector<cudaEvent_t> join;
  cudaEvent_t gjoin = nullptr;
  long pool_tiles = 304;             // pooling threshold in tiles: waves x SMs
  int sms = kSms;
  std::mutex mu;
  std::condition_variable cv;
  struct Req {
    TcPrepared p;
    int member = 0;
    bool released = false;
    cudaEvent_t after = nullptr;
    cudaError_t status = cudaSuccess;
  };
  std::vector<Req*> pending;
  long pending_tiles = 0;
  int live = 0;
  long long launches = 0, pooled_products = 0;
  std::string err;

  // with mu held: launch every pending product and release the posting threads
  void launch_pending() {
    cudaError_t e = cudaSuccess;
    EarlyLaunches none(0);  // behind events of other streams
    for (Req* r : pending)
      if (e == cudaSuccess) e = cudaStreamWaitEvent(gst, ready[r->member], 0);
    std::vector<bool> taken(pending.size(), false);
    for (size_t i = 0; i < pending.size() && e == cudaSuccess; ++i) {
      if (taken[i]) continue;
      const TcPrepared* p[kTcMaxGroup];
      int n = 0;
      for (size_t j = i; j < pending.size() && n < kTcMaxGroup; ++j) {
        if (taken[j] || pending[j]->p.variant != pending[i]->p.variant) continue;
        taken[j] = true;
        p[n++] = &pending[j]->p;
      }
      e = gemm_tc_launch(p, n, gst);
      ++launches;
      pooled_products += n;
    }
    cudaEvent_t ev = done[done_pos++ % done.size()];
    if (e == cudaSuccess) e = cudaEventRecord(ev, gst);
    for (Req* r : pending) {
      r->after = ev;
      r->status = e;
      r->released = true;
    }
    pending.clear();
    pending_tiles = 0;
    cv.notify_all();
  }
};

namespace {

bool group_pools(qtx_rgf_plan_s* P) { return P->group && P->group->pool_tiles > 0; }

cudaError_t group_gemm(qtx_rgf_plan_s* P, const TcArgs& a, int digits, cudaStream_t st) {
  qtx_rgf_group_s* G = P->group;
  qtx_rgf_group_s::Req r;
  r.member = P->member;
  cudaError_t e = gemm_tc_prepare(a, digits, P->ws + P->L.tc_scratch, P->L.tc_bytes, P->d_err_flag, st, &r.p);
  if (e != cudaSuccess || r.p.tiles == 0) return e;
  if (r.p.tiles >= G->pool_tiles) {  // fills the GPU alone (or pooling is off)
    const TcPrepared* one[1] = {&r.p};
    return gemm_tc_launch(one, 1, st);
  }
  if ((e = cudaEventRecord(G->ready[P->member], st)) != cudaSuccess) return e;
  {
    std::unique_lock<std::mutex> lk(G->mu);
    G->pending.push_back(&r);
    G->pending_tiles += r.p.tiles;
    if (G->pending_tiles >= G->pool_tiles || (int)G->pending.size() == G->live) G->launch_pending();
    while (!r.released)
      if (!G->cv.wait_for(lk, std::chrono::microseconds(kPoolWaitUs), [&] { return r.released; }))
        G->launch_pending();
  }
  if (r.status != cudaSuccess) return r.status;
  return cudaStreamWaitEvent(st, r.after, 0);
}

// a member leaves the group when its solve has returned (successfully or not)
void group_leave(qtx_rgf_group_s* G) {
  std::unique_lock<std::mutex> lk(G->mu);
  --G->live;
  if (G->live > 0 && !G->pending.empty() && (int)G->pending.size() == G->live) G->launch_pending();
}

}  // namespace

extern "C" {

qtx_status qtx_rgf_group_create(int n_plans, const qtx_rgf_plan* plans, qtx_rgf_group* out) {
  if (!out || n_plans < 1 || !plans) return QTX_ERR_INVALID_ARG;
  *out = nullptr;
  for (int m = 0; m < n_plans; ++m)
    if (!plans[m] || plans[m]->group) return QTX_ERR_INVALID_ARG;
  auto* G = new qtx_rgf_group_s();
  G->plans.assign(plans, plans + n_plans);
  int dev = 0, sms = kSms;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  G->pool_tiles = (long)kPoolWaves * sms;
  G->sms = sms;
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&G->gst, cudaStreamNonBlocking);
  G->mst.assign(n_plans, nullptr);
  G->ready.assign(n_plans, nullptr);
  G->join.assign(n_plans, nullptr);
  G->done.assign(4, nullptr);
  for (int m = 0; m < n_plans && e == cudaSuccess; ++m) {
    e = cudaStreamCreateWithFlags(&G->mst[m], cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&G->ready[m], cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&G->join[m], cudaEventDisableTiming);
  }
  for (auto& ev : G->done)
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&G->fork, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&G->gjoin, cudaEventDisableTiming);
  if (e != cudaSuccess) {
    g_create_error = std::string("group set-up: ") + cudaGetErrorString(e);
    qtx_rgf_group_destroy(G);
    return QTX_ERR_CUDA;
  }
  *out = G;
  return QTX_OK;
}

qtx_status qtx_rgf_group_solve(qtx_rgf_group G, const qtx_rgf_inputs* const* in, const qtx_rgf_outputs* const* out,
                               void* stream) {
  if (!G || !in || !out) return QTX_ERR_INVALID_ARG;
  const int n = (int)G->plans.size();
  for (int m = 0; m < n; ++m)
    if (!in[m] || !out[m] || !out[m]->status_per_energy) {
      G->err = "group solves need inputs, outputs and a status_per_energy array for every member";
      return QTX_ERR_INVALID_ARG;
    }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  G->err.clear();
  if (cudaEventRecord(G->fork, st) != cudaSuccess) { G->err = "fork event"; return QTX_ERR_CUDA; }
  for (int m = 0; m < n; ++m)
    if (cudaStreamWaitEvent(G->mst[m], G->fork, 0) != cudaSuccess) { G->err = "fork wait"; return QTX_ERR_CUDA; }
  // the group stream starts after the caller's earlier work too
  if (cudaStreamWaitEvent(G->gst, G->fork, 0) != cudaSuccess) { G->err = "fork wait"; return QTX_ERR_CUDA; }
  std::vector<qtx_status> res(n, QTX_OK);
  G->live = n;
  G->pending.clear();
  for (int m = 0; m < n; ++m) {
    G->plans[m]->group = G;
    G->plans[m]->member = m;
  }
  std::vector<std::thread> th;
  th.reserve(n);
  for (int m = 0; m < n; ++m)
    th.emplace_back([&, m] {
      res[m] = qtx_rgf_solve(G->plans[m], in[m], out[m], G->mst[m]);
      group_leave(G);
    });
  for (auto& t : th) t.join();
  for (int m = 0; m < n; ++m) {
    G->plans[m]->group = nullptr;
    G->plans[m]->member = -1;
  }
  qtx_status worst = QTX_OK;
  for (int m = 0; m < n; ++m)
    if (res[m] != QTX_OK && worst == QTX_OK) {
      worst = res[m];
      G->err = std::string("member ") + std::to_string(m) + ": " + G->plans[m]->err;
    }
  // join every member stream and the group stream back into the caller's stream
  for (int m = 0; m < n; ++m) {
    if (cudaEventRecord(G->join[m], G->mst[m]) != cudaSuccess || cudaStreamWaitEvent(st, G->join[m], 0) != cudaSuccess) {
      if (worst == QTX_OK) { worst = QTX_ERR_CUDA; G->err = "join"; }
    }
  }
  if (cudaEventRecord(G->gjoin, G->gst) != cudaSuccess || cudaStreamWaitEvent(st, G->gjoin, 0) != cudaSuccess) {
    if (worst == QTX_OK) { worst = QTX_ERR_CUDA; G->err = "join"; }
  }
  return worst;
}

qtx_status qtx_rgf_group_set_pool_waves(qtx_rgf_group G, int waves) {
  if (!G || waves < 0) return QTX_ERR_INVALID_ARG;
  G->pool_tiles = (long)waves * G->sms;  // 0: every product fills "0 waves", so none is pooled
  return QTX_OK;
}

long long qtx_rgf_group_launches(qtx_rgf_group G) { return G ? G->launches : 0; }

long long qtx_rgf_group_pooled_products(qtx_rgf_group G) { return G ? G->pooled_products : 0; }

const char* qtx_rgf_group_last_error(qtx_rgf_group G) { return G ? G->err.c_str() : g_create_error.c_str(); }

qtx_status qtx_rgf_group_destroy(qtx_rgf_group G) {
  if (!G) return QTX_OK;
  for (auto s : G->mst)
    if (s) cudaStreamDestroy(s);
  if (G->gst) cudaStreamDestroy(G->gst);
  for (auto e : G->ready)
    if (e) cudaEventDestroy(e);
  for (auto e : G->join)
    if (e) cudaEventDestroy(e);
  for (auto e : G->done)
    if (e) cudaEventDestroy(e);
  if (G->fork) cudaEventDestroy(G->fork);
  if (G->gjoin) cudaEventDestroy(G->gjoin);
  delete G;
  return QTX_OK;
}

}  // extern "C"
