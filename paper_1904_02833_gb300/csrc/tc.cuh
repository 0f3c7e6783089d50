// Fifth-generation tensor core (tcgen05) and mbarrier helpers for sm_103a, inline PTX.
//
// Operand tiles live in shared memory in the canonical K-major layout without swizzle:
// the matrix is cut into 8-row x 16-byte "core matrices" (8 x 8 bf16) stored as 128
// contiguous bytes; core matrices adjacent along K are `lbo` bytes apart and 8-row groups
// adjacent along M (or N) are `sbo` bytes apart.  With K elements per row:
//   byte offset of (m, k) = ((m / 8) * (K / 8) + k / 8) * 128 + (m % 8) * 16 + (k % 8) * 2
// i.e. lbo = 128 and sbo = K / 8 * 128.  Accumulators are FP32 in tensor memory: lane m
// of the allocation holds row m, one column per output element.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace snakesim {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Byte offset of element (m, k) of a K-major bf16 tile with K columns.
__device__ __forceinline__ uint32_t kmajor_off(int m, int k, int K) {
  return (uint32_t)((((m >> 3) * (K >> 3) + (k >> 3)) << 7) + ((m & 7) << 4) + ((k & 7) << 1));
}

// Shared-memory matrix descriptor (no swizzle, K-major canonical layout).
__device__ __forceinline__ uint64_t make_sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version of the 5th-generation tensor core
  // base offset 0, absolute-address LBO mode, layout type 0 (no swizzle)
  return d;
}

// The transpose of a K-major tile (above) as an operand: the tile of matrix T [k][n] read
// MN-major, its rows k the reduction dimension, from the 16-row step that starts at saddr.
// A core matrix of the tile (8 rows x 16 bytes along n) is one of the MN-major layout too;
// 8-element groups along n are 128 bytes apart (the stride offset), 8-row groups along k
// `rows8` bytes (the leading offset).
__device__ __forceinline__ uint64_t mn_desc(uint32_t saddr, uint32_t rows8) {
  return make_sdesc(saddr, rows8, 128);
}

// Instruction descriptor of kind::f16 with BF16 A and B, FP32 accumulator; each operand
// K-major, or MN-major where the flag says so.
__host__ __device__ constexpr uint32_t make_idesc_bf16(int M, int N, bool a_mn = false, bool b_mn = false) {
  return (1u << 4)                       // D format: F32
         | (1u << 7)                     // A format: BF16
         | (1u << 10)                    // B format: BF16
         | ((a_mn ? 1u : 0u) << 15)      // A major
         | ((b_mn ? 1u : 0u) << 16)      // B major
         | ((uint32_t)(N >> 3) << 17)    // N / 8
         | ((uint32_t)(M >> 4) << 24);   // M / 16
}

// D[tmem] (+)= A[smem] * B[smem]^T, one elected thread.
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                         uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
      :
      : "r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrive on `mbar` once all previously issued MMAs of this thread have completed.
__device__ __forceinline__ void mma_commit(uint64_t* mbar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
      :
      : "r"(smem_u32(mbar))
      : "memory");
}

// Whole warp: allocate `ncols` TMEM columns (power of two >= 32); address written to *dst.
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
               :
               : "r"(smem_u32(dst)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(ncols)
               : "memory");
}

__device__ __forceinline__ void fence_before_sync() {
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
}
__device__ __forceinline__ void fence_after_sync() {
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
}
// Makes this thread's generic-proxy shared-memory writes visible to the tensor core.
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}

// Warp: 32 consecutive FP32 columns of the warp's 32 TMEM lanes, one lane per thread.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// The same in two steps, N = 16 or 32 columns: the load, then the wait that makes its
// registers valid (they pass through it, so no use of them can move before it).  One load
// may be in flight while the values of another are worked on; the wait is for all of them.
#define TC_R4(r, i) "+r"(r[i]), "+r"(r[i + 1]), "+r"(r[i + 2]), "+r"(r[i + 3])
#define TC_O4(r, i) "=r"(r[i]), "=r"(r[i + 1]), "=r"(r[i + 2]), "=r"(r[i + 3])
__device__ __forceinline__ void tmem_load(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : TC_O4(r, 0), TC_O4(r, 4), TC_O4(r, 8), TC_O4(r, 12), TC_O4(r, 16), TC_O4(r, 20), TC_O4(r, 24), TC_O4(r, 28)
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_load(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : TC_O4(r, 0), TC_O4(r, 4), TC_O4(r, 8), TC_O4(r, 12)
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : TC_R4(r, 0), TC_R4(r, 4), TC_R4(r, 8), TC_R4(r, 12), TC_R4(r, 16), TC_R4(r, 20), TC_R4(r, 24),
                 TC_R4(r, 28)::"memory");
}
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[16], uint32_t (&q)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : TC_R4(r, 0), TC_R4(r, 4), TC_R4(r, 8), TC_R4(r, 12), TC_R4(q, 0), TC_R4(q, 4), TC_R4(q, 8),
                 TC_R4(q, 12)::"memory");
}
#undef TC_R4
#undef TC_O4

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint64_t* mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(mbar)), "r"(count)
               : "memory");
}

// Waits for the phase with parity `parity` to complete, giving up after `limit` polls.
// Returns false on timeout (the caller records an error instead of hanging).
__device__ __forceinline__ bool mbar_wait(uint64_t* mbar, uint32_t parity, uint32_t limit) {
  const uint32_t a = smem_u32(mbar);
  for (uint32_t i = 0; i < limit; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

}  // namespace tc
}  // namespace snakesim
