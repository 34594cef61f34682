// 5th-generation tensor-core building blocks (tcgen05, sm_100-family): TMEM
// allocation, shared-memory operand descriptors for the no-swizzle K-major
// core-matrix layout, BF16 x BF16 -> FP32 MMA issued by one thread, completion
// through an mbarrier with a bounded wait, and TMEM -> register loads.
#pragma once

#include <cstdint>

namespace sas {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Operand layout (K-major, no swizzle): 8-row x 16-byte core matrices; element
// (row, k) of a matrix with kc = K/8 core matrices per row group sits at byte
// ((row/8)*kc + k/8)*128 + (row%8)*16 + (k%8)*2.  Adjacent core matrices along
// K are 128 bytes apart (the descriptor's leading-dimension offset), adjacent
// row groups kc*128 bytes apart (its stride-dimension offset).
__host__ __device__ __forceinline__ uint32_t cm_offset(int row, int k, int kc) {
  return (uint32_t)(((row >> 3) * kc + (k >> 3)) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, int kc) {
  const uint32_t lbo = 128, sbo = (uint32_t)kc * 128;
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// Descriptor with explicit strides (no swizzle, K-major): lbo = bytes between
// core matrices adjacent along K, sbo = bytes between core matrices adjacent
// along M/N.  With sbo = 128 the rows of an operand sit at a uniform 16-byte
// stride, so the operand may start at any row (a shifted window of a larger
// matrix) as long as the address stays 16-byte aligned.
__device__ __forceinline__ uint64_t smem_desc_strided(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16 with BF16 A and B (both K-major) and an
// FP32 accumulator: N/8 at bit 17, M/16 at bit 24.
__host__ __device__ constexpr uint32_t idesc_bf16(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// The same with both operands MN-major (bits 15 and 16): for rows of an operand
// (its M or N index) contiguous in shared memory.  Without swizzle element (mn, k)
// then sits at (mn / 8) * SBO + (k / 8) * LBO + (k % 8) * 16 + (mn % 8) * 2 bytes.
__host__ __device__ constexpr uint32_t idesc_bf16_mn(int m, int n) { return idesc_bf16(m, n) | (1u << 15) | (1u << 16); }

// An FP32 value as two BF16 values (hi, lo) that add up to it after its lowest 13
// mantissa bits are cut -- what kind::tf32 reads of it -- and as three that add up
// to all of it.  Infinities and NaN go to hi alone.
__device__ __forceinline__ void split_tf32(float g, uint16_t& hi, uint16_t& lo) {
  const uint32_t t = __float_as_uint(g) & 0xffffe000u, h = t & 0xffff0000u;
  const float r = __uint_as_float(t) - __uint_as_float(h);
  hi = (uint16_t)(h >> 16);
  lo = (t & 0x7f800000u) == 0x7f800000u ? (uint16_t)0 : (uint16_t)(__float_as_uint(r) >> 16);
}
__device__ __forceinline__ void split_fp32(float g, uint16_t& hi, uint16_t& mid, uint16_t& lo) {
  const uint32_t t = __float_as_uint(g), h = t & 0xffff0000u;
  const bool finite = (t & 0x7f800000u) != 0x7f800000u;
  const float r1 = finite ? g - __uint_as_float(h) : 0.f;
  const uint32_t m = __float_as_uint(r1) & 0xffff0000u;
  const float r2 = r1 - __uint_as_float(m);
  hi = (uint16_t)((h | (finite || !(t & 0xffffu) ? 0u : 0x10000u)) >> 16);  // a NaN stays one
  mid = (uint16_t)(m >> 16);
  lo = (uint16_t)(__float_as_uint(r2) >> 16);
}

// 16 bytes from global to shared memory without a register stop; zeros when !valid
// (the source is not read then).  cp_commit closes a group; cp_wait<N> waits until at
// most N groups of this thread are in flight.
__device__ __forceinline__ void cp16(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// One warp: allocate ncols (power of two >= 32) TMEM columns; base written to *slot.
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(uint32_t base, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(ncols));
}

__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;"); }
// Makes this thread's generic-proxy shared-memory writes visible to the tensor core.
__device__ __forceinline__ void fence_smem_to_async() { asm volatile("fence.proxy.async.shared::cta;"); }

// D[tmem] (+)= A * B^T, M x N x 16, one thread.
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate));
}

// Arrive once on the mbarrier when every MMA this thread issued has completed.
__device__ __forceinline__ void commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

// Waits for the phase with the given parity to complete; gives up after
// max_polls polls (each poll may block briefly in hardware).  Returns true on
// completion.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint32_t max_polls) {
  uint32_t done = 0;
  for (uint32_t i = 0; i < max_polls && !done; ++i) {
    asm volatile(
        "{\n\t.reg .pred P;\n\tmbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\tselp.u32 %0, 1, 0, P;\n\t}\n"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity));
  }
  return done != 0;
}

// 16 consecutive FP32 columns of this thread's TMEM lane (warp w reads lanes
// 32*(w%4) .. 32*(w%4)+31; taddr carries the lane in its upper 16 bits).
__device__ __forceinline__ void ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// 8 consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

}  // namespace tc
}  // namespace sas
