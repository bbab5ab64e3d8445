// Tensor memory and the integer tcgen05 MMA (sm_100a): allocation, 32-lane loads and stores, operand descriptors.
#ifndef DETAG_TENSOR_MEMORY_CUH
#define DETAG_TENSOR_MEMORY_CUH

#include <cuda_runtime.h>

#include <cstdint>

#include "pipeline.cuh"

namespace detag {

namespace {

// One warp; the address goes to `slot` in shared memory.  Waits while another CTA of this SM holds the columns; that
// CTA never depends on this one.
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, unsigned columns) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_addr(slot)), "r"(columns) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}

__device__ __forceinline__ void tmem_free(uint32_t addr, unsigned columns) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(columns));
}

__device__ __forceinline__ void tmem_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_store() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_load() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 32 columns of the calling warp's 32 lanes (lanes 32 (warp % 4) .. + 31, in the address' upper half).
__device__ __forceinline__ void tmem_store32(uint32_t addr, const uint32_t (&w)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(addr),
      "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]), "r"(w[8]), "r"(w[9]),
      "r"(w[10]), "r"(w[11]), "r"(w[12]), "r"(w[13]), "r"(w[14]), "r"(w[15]), "r"(w[16]), "r"(w[17]), "r"(w[18]),
      "r"(w[19]), "r"(w[20]), "r"(w[21]), "r"(w[22]), "r"(w[23]), "r"(w[24]), "r"(w[25]), "r"(w[26]), "r"(w[27]),
      "r"(w[28]), "r"(w[29]), "r"(w[30]), "r"(w[31])
      : "memory");
}

__device__ __forceinline__ void tmem_store8(uint32_t addr, const uint32_t (&w)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr), "r"(w[0]),
               "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}

// Eight columns; the values may be used after tmem_wait_load().
__device__ __forceinline__ void tmem_load8(uint32_t addr, int (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(addr)
               : "memory");
}

// Instruction descriptor of kind::i8: 32-bit integer sums (2 at bit 4), signed bytes for A and B (1 at bits 7 and 10),
// both K-major, N a multiple of 16 up to 256 (N / 8 at bit 17), M = 128 (M / 16 at bit 24).
__host__ __device__ constexpr uint32_t mma_i8_desc(int n) {
  return (2u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n / 8) << 17) | ((128u / 16) << 24);
}

// Descriptor of an operand in shared memory: K-major core matrices of 8 rows x 16 bytes without swizzle, row groups
// `row_stride` bytes apart, the two halves of K `k_stride` bytes apart.  Addresses advance by 16 bytes per unit.
__device__ __forceinline__ uint64_t mma_operand(uint32_t addr, uint32_t row_stride, uint32_t k_stride) {
  return static_cast<uint64_t>((addr & 0x3ffffu) >> 4) | (static_cast<uint64_t>(k_stride >> 4) << 16) |
         (static_cast<uint64_t>(row_stride >> 4) << 32) | (1ull << 46);
}

// D[128][N] (tensor memory) (+)= A[128][32 bytes] (tensor memory) x B[N][32 bytes] (shared memory).  Called by a whole
// warp, issued by the lane whose `leader` is set.
__device__ __forceinline__ void mma_i8(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, unsigned accumulate, bool leader) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "setp.ne.u32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
      "r"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(leader ? 1u : 0u)
      : "memory");
}

// The same with A[128][32 bytes] in shared memory.
__device__ __forceinline__ void mma_i8_shared(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, unsigned accumulate, bool leader) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "setp.ne.u32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(leader ? 1u : 0u)
      : "memory");
}

// The barrier gets one arrival when every MMA the leader has issued so far is complete.
__device__ __forceinline__ void mma_commit(uint64_t* bar, bool leader) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(s_addr(bar)),
      "r"(leader ? 1u : 0u)
      : "memory");
}

}  // namespace

}  // namespace detag
#endif  // DETAG_TENSOR_MEMORY_CUH
