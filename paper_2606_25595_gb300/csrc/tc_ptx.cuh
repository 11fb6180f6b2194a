// Inline-PTX building blocks of the tensor-core kernels (tc_engine.cu, tc_fp64.cu): mbarriers with bounded
// waits, bulk copies, tcgen05 MMA / commit / TMEM loads and the descriptors of their operand tiles.
#pragma once
#include <stdint.h>

namespace qtx {
namespace tc {

constexpr int BM = 128;        // output rows per CTA (TMEM lanes)
constexpr int BKS = 16;        // bf16 K elements per stage (32-byte rows, 32B swizzle) = one MMA K
constexpr int TILE_A = BM * BKS * 2;   // bytes of one A-plane tile (128 rows x 32 B)
constexpr int DW = 7;          // bits per digit below the leading one

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(su32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait: gives up after limit_ns of %globaltimer (2 s in normal launches), raising *err, or as
// soon as another thread has raised it.
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, int* err, uint64_t limit_ns) {
  if (mbar_try(b, parity)) return true;
  const uint64_t t0 = gtimer();
  while (true) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try(b, parity)) return true;
    if (*((volatile int*)err)) return false;
    if (gtimer() - t0 > limit_ns) {
      atomicExch(err, 1);
      return false;
    }
    __nanosleep(128);
  }
}
// Bounded wait for work this CTA has already issued (bulk copies, MMAs) to complete, used on the way
// out after an error: it does not give up because *err is raised, only after limit_ns.
__device__ __forceinline__ bool mbar_wait_drain(uint64_t* b, uint32_t parity, uint64_t limit_ns) {
  const uint64_t t0 = gtimer();
  while (!mbar_try(b, parity)) {
    if (gtimer() - t0 > limit_ns) return false;
    __nanosleep(64);
  }
  return true;
}
constexpr uint64_t kWaitLimitNs = 2000000000ull;   // bounded waits of normal launches
constexpr uint64_t kWaitTestLimitNs = 100000ull;   // with the wait test switched on
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(su32(dst)), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(su32(bar))
      : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major, 32-byte swizzle, 8-row groups 256 bytes apart.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1u << 16;            // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(256u >> 4) << 32;   // stride byte offset
  d |= (uint64_t)1u << 46;            // descriptor version for tcgen05
  d |= (uint64_t)6u << 61;            // 32-byte swizzle
  return d;
}
// Byte offset of element (row rr, k) inside a K-major tile with 32-byte rows and 32-byte swizzle:
// the 16-byte half-row index is XORed with bit 2 of the row (address bit 4 ^= address bit 7).
__host__ __device__ __forceinline__ uint32_t sw32_offset(uint32_t rr, uint32_t kk) {
  const uint32_t o = rr * 32u + kk * 2u;
  return o ^ (((o >> 7) & 1u) << 4);
}
// Instruction descriptor: kind::f16, D = F32, A = B = BF16, both K-major, M = 128, N = n (a multiple
// of 16, up to 128 here).
__host__ __device__ constexpr uint32_t idesc_n(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

__device__ __forceinline__ void mma(uint32_t dtmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(dtmem), "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Tile of round k for this CTA.  Round k covers tiles [k G, (k + 1) G) (G = gridDim.x; column tile
// fastest, then row tile, then batch entry), dealt to the CTAs rotated by one per round: the
// narrower last column tile then falls to every CTA equally often (whenever G - 1 is coprime to the
// number of column tiles, always for 152 SMs) rather than to a fixed subset of them, while the
// tiles in flight at any time stay those of a few neighbouring batch entries, which share operands
// through L2.
__device__ __forceinline__ long tile_at(int k) {
  const int G = (int)gridDim.x;
  int b = (int)blockIdx.x - k % G;
  if (b < 0) b += G;
  return (long)k * G + b;
}

}  // namespace tc
}  // namespace qtx
