// FPX storage codec (Sec. V: byte-aligned custom floating-point formats FPX, X in {56, 48, 40, 32,
// 24, 16} bits = sign + the 8-bit exponent of FP32 (bias 127) + X - 9 significand bits, written
// with IEEE-754 rounding so that FP32 is one of them bit for bit; Sec. III: a value cutoff below
// which magnitudes are stored as zero).
//
// Rounding is to nearest, ties to even, from the FP64 value; results beyond the largest finite
// value become +-inf, values below 2^-126 become FP32-style subnormals (exponent field 0, value
// q 2^(-126-m)); NaN is stored as the quiet NaN code, infinities stay infinite, a result that
// rounds to zero keeps its sign, and the cutoff gives +0.  A stream of n values is the
// concatenation of their X/8-byte little-endian codes.
//
// Kernels: one thread per group of 8 values, whose X bytes are X/8 aligned 64-bit words (the codes of
// the group laid end to end).  The plan uses the same kernels on its own sweep types (FP64, FP32 and df32 values, converted exactly to FP64 first) to keep the
// left-connected blocks compressed between the forward and the backward sweeps.
#include <type_traits>

#include "../../include/qtx_kernels.h"
#include "df32.cuh"
#include "kernels.cuh"

namespace qtx {
namespace {

// the general case: specials, zeros, subnormal results and magnitudes below the cutoff
template <int BITS>
__device__ __noinline__ uint64_t fpx_encode_rare(double x, double cutoff) {
  constexpr int m = BITS - 9;
  const uint64_t u = (uint64_t)__double_as_longlong(x);
  const uint64_t s = u >> 63;
  const int e = (int)((u >> 52) & 0x7FF);
  const uint64_t f = u & ((1ull << 52) - 1);
  if (e == 0x7FF) {  // infinity or NaN
    if (f) return (0xFFull << m) | (1ull << (m - 1));
    return (s << (BITS - 1)) | (0xFFull << m);
  }
  // magnitudes order like their bits
  if ((u & 0x7fffffffffffffffull) < (uint64_t)__double_as_longlong(cutoff)) return 0;
  if (e == 0) return s << (BITS - 1);  // FP64 zero or subnormal: far below the smallest FPX value
  const int E = e - 1023 + 127;       // FPX biased exponent of the value
  const uint64_t F = (1ull << 52) | f;
  // q = F >> sh rounded to nearest even; sh = 52 - m for normal results, more for subnormal ones
  const int sh = E >= 1 ? 52 - m : 53 - m - E;
  uint64_t q;
  if (sh >= 64) {
    q = 0;
  } else {
    q = F >> sh;
    const uint64_t rem = F & ((1ull << sh) - 1), half = 1ull << (sh - 1);
    if (rem > half || (rem == half && (q & 1ull))) ++q;
  }
  // normal: q in [2^m, 2^(m+1)]; field = (E << m) + (q - 2^m) carries into the exponent on
  // round-up.  subnormal: field = q (q = 2^m becomes the smallest normal by itself).
  uint64_t field = E >= 1 ? ((uint64_t)E << m) + (q - (1ull << m)) : q;
  if (field >= (0xFFull << m)) field = 0xFFull << m;  // overflow to infinity
  return (s << (BITS - 1)) | field;
}

template <int BITS>
__device__ __forceinline__ uint64_t fpx_encode(double x, double cutoff) {
  constexpr int m = BITS - 9, sh = 52 - m;
  const uint64_t u = (uint64_t)__double_as_longlong(x), v = u & 0x7fffffffffffffffull;
  const uint32_t e = (uint32_t)(v >> 52);
  // normal results: exponent and significand rounded as one integer (ties to even; a carry moves on into
  // the exponent), rebiased; magnitudes order like their bits
  if (e < 1023 - 126 || e == 0x7ff || v < (uint64_t)__double_as_longlong(cutoff)) return fpx_encode_rare<BITS>(x, cutoff);
  const uint64_t r = (v + (((uint64_t)1 << (sh - 1)) - 1) + ((v >> sh) & 1)) >> sh;
  const uint64_t field = r - ((uint64_t)(1023 - 127) << m), inf = (uint64_t)0xFF << m;
  return ((u >> 63) << (BITS - 1)) | (field < inf ? field : inf);
}

template <int BITS>
__device__ __forceinline__ double fpx_decode(uint64_t c) {
  constexpr int m = BITS - 9;
  const uint64_t s = (c >> (BITS - 1)) & 1ull;
  const int ef = (int)((c >> m) & 0xFF);
  const uint64_t q = c & ((1ull << m) - 1);
  uint64_t u;
  if (ef == 0xFF) {
    u = (s << 63) | (0x7FFull << 52) | (q ? (1ull << 51) : 0ull);
  } else if (ef == 0) {
    // q 2^(-126 - m): an FP64 normal number (q < 2^47), its leading bit at position p
    const int p = 63 - __clzll((long long)(q | 1));
    u = (s << 63) | (q ? ((uint64_t)(p - 126 - m + 1023) << 52) | ((q << (52 - p)) & ((1ull << 52) - 1)) : 0ull);
  } else {
    u = (s << 63) | ((uint64_t)(ef - 127 + 1023) << 52) | (q << (52 - m));
  }
  return __longlong_as_double((long long)u);
}

// One block codes 2048 reals (256 groups of 8).  A thread's group is 64 consecutive bytes of FP64 and X
// bytes of codes, so reading and writing it directly touches 32 separate lines a warp and instruction;
// both sides pass through shared memory instead (skewed: thread-wise and warp-wise accesses fall in
// distinct banks), and global accesses are whole lines.  The
// rounding, the cutoff and the conversions of df32 values are integer operations (the FP64 pipe is 1/64 as fast).
// 60 million FP64 values to 24 bits and back: 406 us with direct accesses and FP64 compares, 235 us so.
constexpr int kT = 256, kTile = 8 * kT;
__host__ __device__ constexpr int skew(int k) { return k + (k >> 3); }

template <int BITS, typename T>
__global__ void __launch_bounds__(kT) k_fpx_compress(const T* x, long n, double cutoff, uint64_t* out) {
  constexpr int W = BITS / 8, LD = W | 1;  // 64-bit words per group of 8 codes
  __shared__ T s_x[skew(kTile)];
  __shared__ uint64_t s_w[kT * LD];
  const long k0 = (long)blockIdx.x * kTile;
  const int t = threadIdx.x, m = (int)(n - k0 < kTile ? n - k0 : kTile);
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (t + kT * j < m) s_x[skew(t + kT * j)] = x[k0 + t + kT * j];
  __syncthreads();
  const int groups = (m + 7) / 8;
  if (t < groups) {
    uint64_t w[W];
#pragma unroll
    for (int i = 0; i < W; ++i) w[i] = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint64_t c = 8 * t + j < m ? fpx_encode<BITS>(to_d(s_x[skew(8 * t + j)]), cutoff) : 0ull;
      const int bit = j * BITS, wi = bit / 64, off = bit % 64;
      w[wi] |= c << off;
      if (off + BITS > 64) w[wi + 1] |= c >> (64 - off);
    }
#pragma unroll
    for (int i = 0; i < W; ++i) s_w[t * LD + i] = w[i];
  }
  __syncthreads();
  uint64_t* o = out + (long)blockIdx.x * kT * W;
#pragma unroll
  for (int i = 0; i < W; ++i) {
    const int q = t + kT * i;
    if (q < groups * W) o[q] = s_w[q / W * LD + q % W];
  }
}

template <int BITS, typename T>
__global__ void __launch_bounds__(kT) k_fpx_decompress(const uint64_t* in, long n, T* x) {
  constexpr int W = BITS / 8, LD = W | 1;
  constexpr uint64_t MASK = (1ull << BITS) - 1;
  __shared__ T s_x[skew(kTile)];
  __shared__ uint64_t s_w[kT * LD];
  const long k0 = (long)blockIdx.x * kTile;
  const int t = threadIdx.x, m = (int)(n - k0 < kTile ? n - k0 : kTile), groups = (m + 7) / 8;
  const uint64_t* src = in + (long)blockIdx.x * kT * W;
#pragma unroll
  for (int i = 0; i < W; ++i) {
    const int q = t + kT * i;
    if (q < groups * W) s_w[q / W * LD + q % W] = src[q];
  }
  __syncthreads();
  if (t < groups) {
    uint64_t w[W];
#pragma unroll
    for (int i = 0; i < W; ++i) w[i] = s_w[t * LD + i];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int bit = j * BITS, wi = bit / 64, off = bit % 64;
      uint64_t c = w[wi] >> off;
      if (off + BITS > 64) c |= w[wi + 1] << (64 - off);
      s_x[skew(8 * t + j)] = from_d<T>(fpx_decode<BITS>(c & MASK));
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (t + kT * j < m) x[k0 + t + kT * j] = s_x[skew(t + kT * j)];
}

template <typename T>
cudaError_t launch_compress(int bits, const T* x, long n, double cutoff, void* out, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((n + kTile - 1) / kTile);
  uint64_t* o = reinterpret_cast<uint64_t*>(out);
  switch (bits) {
    case 56: k_fpx_compress<56, T><<<blocks, 256, 0, st>>>(x, n, cutoff, o); break;
    case 48: k_fpx_compress<48, T><<<blocks, 256, 0, st>>>(x, n, cutoff, o); break;
    case 40: k_fpx_compress<40, T><<<blocks, 256, 0, st>>>(x, n, cutoff, o); break;
    case 32: k_fpx_compress<32, T><<<blocks, 256, 0, st>>>(x, n, cutoff, o); break;
    case 24: k_fpx_compress<24, T><<<blocks, 256, 0, st>>>(x, n, cutoff, o); break;
    case 16: k_fpx_compress<16, T><<<blocks, 256, 0, st>>>(x, n, cutoff, o); break;
    default: return cudaErrorInvalidValue;
  }
  count_launch();
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_decompress(int bits, const void* in, long n, T* x, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((n + kTile - 1) / kTile);
  const uint64_t* i = reinterpret_cast<const uint64_t*>(in);
  switch (bits) {
    case 56: k_fpx_decompress<56, T><<<blocks, 256, 0, st>>>(i, n, x); break;
    case 48: k_fpx_decompress<48, T><<<blocks, 256, 0, st>>>(i, n, x); break;
    case 40: k_fpx_decompress<40, T><<<blocks, 256, 0, st>>>(i, n, x); break;
    case 32: k_fpx_decompress<32, T><<<blocks, 256, 0, st>>>(i, n, x); break;
    case 24: k_fpx_decompress<24, T><<<blocks, 256, 0, st>>>(i, n, x); break;
    case 16: k_fpx_decompress<16, T><<<blocks, 256, 0, st>>>(i, n, x); break;
    default: return cudaErrorInvalidValue;
  }
  count_launch();
  return cudaGetLastError();
}

}  // namespace

bool fpx_width_ok(int bits) {
  return bits == 56 || bits == 48 || bits == 40 || bits == 32 || bits == 24 || bits == 16;
}
size_t fpx_bytes(int bits, long n_reals) { return n_reals <= 0 ? 0 : (size_t)((n_reals + 7) / 8) * (size_t)bits; }

template <typename T>
cudaError_t fpx_store(int bits, const cx<T>* x, long n_complex, void* out, cudaStream_t st) {
  return launch_compress<T>(bits, reinterpret_cast<const T*>(x), 2 * n_complex, 0.0, out, st);
}
template <typename T>
cudaError_t fpx_load(int bits, const void* in, long n_complex, cx<T>* x, cudaStream_t st) {
  return launch_decompress<T>(bits, in, 2 * n_complex, reinterpret_cast<T*>(x), st);
}
template cudaError_t fpx_store<double>(int, const cx<double>*, long, void*, cudaStream_t);
template cudaError_t fpx_store<float>(int, const cx<float>*, long, void*, cudaStream_t);
template cudaError_t fpx_store<df>(int, const cx<df>*, long, void*, cudaStream_t);
template cudaError_t fpx_load<double>(int, const void*, long, cx<double>*, cudaStream_t);
template cudaError_t fpx_load<float>(int, const void*, long, cx<float>*, cudaStream_t);
template cudaError_t fpx_load<df>(int, const void*, long, cx<df>*, cudaStream_t);

}  // namespace qtx

using namespace qtx;

extern "C" {

size_t qtx_fpx_bytes(int bits, long n) { return fpx_width_ok(bits) ? fpx_bytes(bits, n) : 0; }

qtx_status qtx_fpx_compress(int bits, const double* x, long n, double cutoff, void* out, void* stream) {
  if (!fpx_width_ok(bits) || n < 0 || !(cutoff >= 0.0)) return QTX_ERR_INVALID_ARG;
  if (n == 0) return QTX_OK;
  if (!x || !out || (reinterpret_cast<uintptr_t>(x) & 7) || (reinterpret_cast<uintptr_t>(out) & 7))
    return QTX_ERR_INVALID_ARG;
  // (the kernel compares bit patterns: a cutoff of -0.0 is none, like 0.0)
  if (cutoff == 0.0) cutoff = 0.0;
  const cudaError_t e = launch_compress<double>(bits, x, n, cutoff, out, reinterpret_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? QTX_OK : QTX_ERR_CUDA;
}

qtx_status qtx_fpx_decompress(int bits, const void* in, long n, double* x, void* stream) {
  if (!fpx_width_ok(bits) || n < 0) return QTX_ERR_INVALID_ARG;
  if (n == 0) return QTX_OK;
  if (!x || !in || (reinterpret_cast<uintptr_t>(x) & 7) || (reinterpret_cast<uintptr_t>(in) & 7))
    return QTX_ERR_INVALID_ARG;
  const cudaError_t e = launch_decompress<double>(bits, in, n, x, reinterpret_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? QTX_OK : QTX_ERR_CUDA;
}

}  // extern "C"
