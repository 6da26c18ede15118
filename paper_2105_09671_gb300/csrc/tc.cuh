// 5th-generation tensor-core (tcgen05) helpers for sm_100-family GPUs:
// tensor-memory allocation, shared-memory matrix descriptors, the BF16 MMA
// with FP32 accumulation in tensor memory, completion through an mbarrier,
// and tensor-memory loads for the epilogue.
//
// Operands are staged by the CTA's threads in the canonical K-major layout
// without swizzle: 8 x 16-byte "core matrices" (8 rows of 8 BF16 along K),
// stored as [row group g][K chunk c][row r][8 elements]; the byte distance
// between K-adjacent core matrices is the leading-dimension offset (LBO) and
// between row groups the stride-dimension offset (SBO).
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"

namespace ac {

// Shared-memory matrix descriptor (64 bit): start address >> 4 in bits 0-13,
// LBO >> 4 in bits 16-29, SBO >> 4 in bits 32-45, the fixed value 1 in bits
// 46-48, base offset 0, no swizzle (bits 61-63 = 0).
__device__ __forceinline__ uint64_t tc_smem_desc(const void *start, uint32_t lbo_bytes,
                                                  uint32_t sbo_bytes) {
  const uint32_t a = smem_u32(start);
  uint64_t d = 0;
  d |= (uint64_t)((a & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// The same for operands in the 64-byte swizzle (layout code 4 in bits 61-63):
// rows of 64 bytes whose 16-byte chunk index is XORed with bits 7-8 of the
// shared-memory address, as TMA's SWIZZLE_64B writes them.  The pattern is
// tied to the address, so a start that is any whole number of rows in (a
// pixel shift) or 32 bytes in (the second half of K) needs base offset 0.
__device__ __forceinline__ uint64_t tc_smem_desc_sw64(const void *start, uint32_t lbo_bytes,
                                                       uint32_t sbo_bytes) {
  return tc_smem_desc(start, lbo_bytes, sbo_bytes) | ((uint64_t)4 << 61);
}

// Instruction descriptor of kind::f16 for BF16 x BF16 -> FP32, both operands
// K-major: D format (bits 4-5) = 1 (F32), A format (7-9) = 1 (BF16), B format
// (10-12) = 1 (BF16), N >> 3 in bits 17-22, M >> 4 in bits 24-28.
__host__ __device__ constexpr uint32_t tc_idesc_bf16_f32(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

// Tensor-memory allocation: one whole warp; writes the base address to *slot.
__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(slot)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// D[tmem] (+)= A[smem] * B[smem]^T, one instruction (M x N x 16), issued by
// one thread.
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                            uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"((uint32_t)accumulate)
      : "memory");
}
// Arrive once on `bar` when every MMA issued before by this thread is done.
__device__ __forceinline__ void tc_commit(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

// 32 consecutive FP32 columns of this thread's tensor-memory lane (the warp
// reads lanes 32 * (warp % 4) .. +31; taddr carries the lane in bits 16-31).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float *v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Byte offset of element (row, k) in a canonical K-major tile with kc K chunks
// of 8 elements per row group: [row/8][k/8][row%8][k%8].
__host__ __device__ __forceinline__ uint32_t tc_kmajor_off(int row, int k, int kc) {
  return (uint32_t)((((row >> 3) * kc + (k >> 3)) * 64 + (row & 7) * 8 + (k & 7)) * 2);
}

}  // namespace ac
