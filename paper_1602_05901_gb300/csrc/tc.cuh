// Inline-PTX wrappers for the Blackwell tensor-core path (sm_103a): mbarriers,
// TMA tensor copies, tcgen05 MMA with accumulators in tensor memory (TMEM).
//
// Conventions used by every kernel that includes this header:
// * Operands are K-major BF16 tiles written by TMA with 128-byte (or 64-byte)
//   swizzling into 1024-byte aligned shared memory: row r of a tile holds the
//   K values of one M (or N) index, 8 rows form one swizzle atom.
// * One elected thread issues all MMAs of a CTA (cta_group::1, M = 128); the
//   accumulator occupies TMEM lanes 0..127 (one lane per M row) and N
//   consecutive 32-bit columns.
// * Every wait is bounded by a deadline on the global timer; a caller that
//   sees a wait give up records an error status and winds down.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace rsv {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t now_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// ---------------------------------------------------------------- mbarriers
__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t *bar, unsigned parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Wait until the phase with the given parity has completed, or the deadline passes.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity, uint64_t deadline) {
    if (mbar_test(bar, parity)) return true;
    while (true) {
        if (mbar_test(bar, parity)) return true;
        if (now_ns() > deadline) return false;
    }
}

// ---------------------------------------------------------------- TMA tensor loads
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int c0, int c1, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_u32(dst)),
        "l"(map), "r"(c0), "r"(c1), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int c0, int c1, int c2, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::
            "r"(smem_u32(dst)),
        "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                            uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(smem_u32(dst)),
        "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void tma_load_5d(void *dst, const CUtensorMap *map, int c0, int c1, int c2, int c3, int c4,
                                            uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, "
        "%6}], [%7];" ::"r"(smem_u32(dst)),
        "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap *map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

// ---------------------------------------------------------------- tcgen05
__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols) {  // whole warp
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {  // whole warp
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor of a K-major, swizzled operand tile.
// swz = 128: rows of 128 B, 8-row atoms of 1024 B; swz = 64: rows of 64 B, atoms of 512 B.
// Fields: start address >> 4 (bits 0-13), leading offset (16-29, unused for
// swizzled K-major), stride between 8-row groups >> 4 (32-45), descriptor
// version 1 (46-47), layout type (61-63: 2 = 128-byte swizzle, 4 = 64-byte).
__device__ __forceinline__ uint64_t kmajor_desc(uint32_t saddr, int swz) {
    const uint64_t sbo = (swz == 128 ? 1024u : 512u) >> 4;
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | (sbo << 32) | ((uint64_t)1 << 46) |
           ((uint64_t)(swz == 128 ? 2 : 4) << 61);
}

// Shared-memory matrix descriptor of an MN-major, swizzled operand tile: each
// row (one K index) holds 64 (128-byte swizzle) or 32 (64-byte swizzle)
// consecutive M/N elements; 8 rows form one swizzle atom (grp bytes apart
// along K: stride offset), and atoms along M/N sit col bytes apart (leading
// offset).
__device__ __forceinline__ uint64_t mnmajor_desc(uint32_t saddr, int swz, uint32_t col, uint32_t grp) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((col >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((grp >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46) | ((uint64_t)(swz == 128 ? 2 : 4) << 61);
}

// Instruction descriptor of kind::f16 with BF16 A and B, FP32 accumulator,
// shape M x N; operands K-major unless a_mn / b_mn (bits 15 and 16).
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool a_mn = false, bool b_mn = false) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// D[tmem] (+)= A[smem] * B[smem]^T for one K = 16 slice.
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
            tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// The same with the descriptors' words apart: operands of one layout differ in the low word only, by their distance
// in 16-byte units.  One thread issues all MMAs, so the instructions between two of them count: rebuilding
// descriptors per MMA took 140 cycles, one addition each in a lone lane 118, in a warp in step 75; the MMAs themselves
// take 46, 53, 61, 69, 102 and 133 cycles for N = 32, 64, 96, 128, 192 and 256 (M = 128, either major order, either
// swizzle).
// For a whole warp in step: `lead` is set in the one lane that issues (elect_one).  The addresses are the same in all
// lanes, so that the compiler can keep them in uniform registers, where the instruction takes its operands from.
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t r;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(r));
    return r;
}
__device__ __forceinline__ void mma_bf16(uint32_t lead, uint32_t tmem_d, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi,
                                         uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p, l;\n .reg .b64 a, b;\n setp.ne.b32 p, %6, 0;\n setp.ne.b32 l, %7, 0;\n mov.b64 a, {%1, %2};\n"
        " mov.b64 b, {%3, %4};\n @l tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}" ::"r"(tmem_d),
        "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(accumulate), "r"(lead)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t lead, uint64_t *bar) {
    asm volatile(
        "{\n .reg .pred l;\n setp.ne.b32 l, %1, 0;\n"
        " @l tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(smem_u32(bar)), "r"(lead)
        : "memory");
}
// The wait of a whole warp in step: the same answer in all lanes.
__device__ __forceinline__ bool warp_wait(uint64_t *bar, unsigned parity, uint64_t deadline) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, deadline));
}
// The mbarrier receives one arrival once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// 16 consecutive FP32 columns of the warp's 32 TMEM lanes: lane l of the warp gets row (lane base + l).
// The values are there after tmem_ld_wait(); tmem_landed, called behind it on the registers of every such load, keeps
// the compiler from moving their uses ahead of the wait (nothing else in the code ties the two together).
__device__ __forceinline__ void tmem_ld16_start(uint32_t taddr, uint32_t r[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_landed(uint32_t r[16]) {
    asm volatile(""
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                   "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]));
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16]) {
    uint32_t r[16];
    tmem_ld16_start(taddr, r);
    tmem_ld_wait();
    tmem_landed(r);
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__host__ __device__ constexpr uint32_t tmem_cols_for(int n) {
    return n <= 32 ? 32u : n <= 64 ? 64u : n <= 128 ? 128u : n <= 256 ? 256u : 512u;
}

}  // namespace tc
}  // namespace rsv
