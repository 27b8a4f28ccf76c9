// tcgen05 (5th-generation tensor core) wrappers shared by the kernels that use tensor memory: matrix descriptors,
// the MMA with its first operand in shared or in tensor memory, commits, tensor-memory loads and stores, tiled TMA boxes.
#pragma once

#include <cuda.h>

#include "spla_device.cuh"

namespace spla {

// Instruction descriptor, kind::f16 with fp32 accumulators (bit 4): operand types at bits 7 (A) and 10 (B), 0 = fp16,
// 1 = bf16 (both operands always have the same type); majorness at bits 15 (A) and 16 (B), 1 = MN-major; N / 8 at bit
// 17, M / 16 at bit 24.
__host__ __device__ constexpr uint32_t umma_idesc(bool bf16, bool a_mn, bool b_mn, int M, int N) {
  return (1u << 4) | (bf16 ? (1u << 7) | (1u << 10) : 0u) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
         ((uint32_t)(N / 8) << 17) | ((uint32_t)(M / 16) << 24);
}

// Shared-memory matrix descriptor of an operand stored as rows of 128 bytes with the 128-byte swizzle (atoms of 8 rows,
// 1024-byte aligned): start address / 16, leading byte offset / 16 at bit 16, stride byte offset (between groups of 8
// rows) / 16 at bit 32, descriptor version 1 at bit 46, layout type 2 at bit 61.
//   K-major operand  (a row holds 64 consecutive k of one m / n):  the leading offset is not used; the next 16 k are 32
//                    bytes further inside the row, the next 64 in the next array of rows;
//   MN-major operand (a row holds 64 consecutive m / n of one k):  the leading offset is the distance between the arrays
//                    of rows that hold neighbouring groups of 64 m / n; the next 16 k are 16 rows = 2048 bytes further.
// In two words, for loops that step through an operand: the low word grows by bytes / 16 (shared memory ends below the 18
// bits that the address field covers, so it never carries), the high word is the same for all.
constexpr uint32_t kUmmaDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t umma_desc_lo(uint32_t smem_addr, uint32_t lead_bytes) { return (smem_addr >> 4) | ((lead_bytes >> 4) << 16); }
__device__ __forceinline__ uint64_t umma_desc_of(uint32_t lo) { return ((uint64_t)kUmmaDescHi << 32) | lo; }

// D (tensor memory) (+)= A B, A and B in shared memory; for a whole warp whose lanes all hold the operands, `one` non-zero
// in the lane that issues.  Operands that are the same in every lane of a converged warp can stay in uniform registers;
// issued from a branch that only one lane takes, an MMA cost 75 to 110 cycles in a loop beside busy warps, this way 50 to 65.
__device__ __forceinline__ void umma_ss_one(uint32_t one, uint32_t tmem_d, uint64_t desc_a, uint64_t desc_b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.ne.b32 q, %6, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5}, p;\n\t}"
      ::"r"(tmem_d), "l"(desc_a), "l"(desc_b), "r"(idesc), "r"(accumulate), "r"(0u), "r"(one)
      : "memory");
}
// Four k-steps in one go (the predicates are formed once): D (+)= A B + three more that always accumulate.  DA, DB: what the
// low descriptor words grow by per step.
template <uint32_t DA, uint32_t DB>
__device__ __forceinline__ void umma_ss4_one(uint32_t one, uint32_t tmem_d, uint32_t lo_a, uint32_t lo_b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %10, 0;\n\t"
      "setp.ne.b32 q, %12, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %5, %9, {%11, %11, %11, %11}, p;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %2, %6, %9, {%11, %11, %11, %11}, 1;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %3, %7, %9, {%11, %11, %11, %11}, 1;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %4, %8, %9, {%11, %11, %11, %11}, 1;\n\t}"
      ::"r"(tmem_d), "l"(umma_desc_of(lo_a)), "l"(umma_desc_of(lo_a + DA)), "l"(umma_desc_of(lo_a + 2 * DA)), "l"(umma_desc_of(lo_a + 3 * DA)),
        "l"(umma_desc_of(lo_b)), "l"(umma_desc_of(lo_b + DB)), "l"(umma_desc_of(lo_b + 2 * DB)), "l"(umma_desc_of(lo_b + 3 * DB)),
        "r"(idesc), "r"(accumulate), "r"(0u), "r"(one)
      : "memory");
}
// ... with A in tensor memory (row m in lane m, two 16-bit k per 32-bit column), DA columns further per step.
template <uint32_t DA, uint32_t DB>
__device__ __forceinline__ void umma_ts4_one(uint32_t one, uint32_t tmem_d, uint32_t tmem_a, uint32_t lo_b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %10, 0;\n\t"
      "setp.ne.b32 q, %12, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %5, %9, {%11, %11, %11, %11}, p;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%2], %6, %9, {%11, %11, %11, %11}, 1;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%3], %7, %9, {%11, %11, %11, %11}, 1;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%4], %8, %9, {%11, %11, %11, %11}, 1;\n\t}"
      ::"r"(tmem_d), "r"(tmem_a), "r"(tmem_a + DA), "r"(tmem_a + 2 * DA), "r"(tmem_a + 3 * DA),
        "l"(umma_desc_of(lo_b)), "l"(umma_desc_of(lo_b + DB)), "l"(umma_desc_of(lo_b + 2 * DB)), "l"(umma_desc_of(lo_b + 3 * DB)),
        "r"(idesc), "r"(accumulate), "r"(0u), "r"(one)
      : "memory");
}
// Arrives on the barrier once every tcgen05.mma issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit_one(uint32_t one, uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(bar)), "r"(one)
      : "memory");
}
// One lane of a converged warp.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b32 d;\n\t"
      "elect.sync d|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r));
  return r;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// One warp, all lanes: allocates `cols` tensor-memory columns (a power of two >= 32), the base address goes to *out.
__device__ __forceinline__ void tmem_alloc(uint32_t* out, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(out)), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t base, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols) : "memory");
}

// 32 consecutive columns of this thread's tensor-memory lane.  tmem_ld_wait32() before the values are used.
__device__ __forceinline__ void tmem_ld32_async(uint32_t addr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(addr)
      : "memory");
}
// (the registers pass through the wait, so that no use of them can be moved before it)
__device__ __forceinline__ void tmem_ld_wait32(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                 "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                 "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :: "memory");
}
__device__ __forceinline__ void tmem_ld16_async(uint32_t addr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                 "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait16(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :: "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t addr, float (&v)[32]) {
  uint32_t r[32];
  tmem_ld32_async(addr, r);
  tmem_ld_wait32(r);
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
// 16 consecutive columns of this thread's lane written; tmem_st_wait() before anybody is told.
__device__ __forceinline__ void tmem_st16(uint32_t addr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// One TMA box of a two-dimensional map (never multicast).
__device__ __forceinline__ void tma_load_box(uint32_t dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
               "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void mbar_arrive1(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Warp-uniform bounded waits of kernels with roles: every lane of a warp goes on, or every lane gives up (the tensor-memory
// instructions want whole warps).  `limit` as for mbar_wait.
__device__ __forceinline__ bool warp_waits(uint64_t* bar, uint32_t parity, int limit) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, limit));
}
__device__ __forceinline__ bool warp_aborted(volatile int* flag) { return __any_sync(0xffffffffu, *flag != 0); }
// Generic-proxy accesses to shared memory before this are ordered before asynchronous-proxy ones (TMA, tensor core) after it.
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

}  // namespace spla
