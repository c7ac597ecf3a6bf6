// tcgen05 / TMEM building blocks for sm_103a (inline PTX).
//
// Shared-memory operand layout: K-major, 64-byte swizzle.  A tile of R rows x 64 bytes of K is
// stored row after row; rows are grouped by 8 into 512-byte atoms (tile base 512-byte aligned),
// and the 16-byte chunk c of row r sits at chunk position c ^ ((r / 2) % 4).
//
// Every wait in here is bounded: a wait that runs out returns false, which its caller reports.
#pragma once

#include <cuda_bf16.h>
#include <cstdint>

namespace lg {
namespace tc {

constexpr long long kSpinLimit = 1LL << 21;   // polls of one wait: about 8 s (the hardware suspends each for 4 us)

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor for a 64-byte-swizzled K-major tile: stride between
// 8-row groups 512 bytes, descriptor version 1, swizzle mode 4 (64 bytes).
__host__ __device__ constexpr uint64_t make_desc_sw64(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)1u << 16;
    d |= (uint64_t)(512u >> 4) << 32;
    d |= (uint64_t)1u << 46;
    d |= (uint64_t)4u << 61;
    return d;
}

// Instruction descriptor, kind::f16: bf16 x bf16 -> f32, both operands K-major, M x N.
__host__ __device__ constexpr uint32_t make_idesc_bf16(int M, int N) {
    return (1u << 4)                       // D format: f32
           | (1u << 7)                     // A format: bf16
           | (1u << 10)                    // B format: bf16
           | ((uint32_t)(N >> 3) << 17)    // N / 8
           | ((uint32_t)(M >> 4) << 24);   // M / 16
}

// Instruction descriptor, kind::tf32: tf32 x tf32 -> f32, both operands K-major, M x N.
__host__ __device__ constexpr uint32_t make_idesc_tf32(int M, int N) {
    return (1u << 4)                       // D format: f32
           | (2u << 7)                     // A format: tf32
           | (2u << 10)                    // B format: tf32
           | ((uint32_t)(N >> 3) << 17)    // N / 8
           | ((uint32_t)(M >> 4) << 24);   // M / 16
}

// Round an FP32 value to TF32 (round to nearest, ties away); result in an FP32 container.
__device__ __forceinline__ float to_tf32(float x) {
    uint32_t u;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(x));
    return __uint_as_float(u);
}

__device__ __forceinline__ void tmem_alloc(uint32_t *dst_smem, int ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, int ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---- issue by a whole warp
// The operands of tcgen05.mma are uniform registers.  Code that runs in one thread of a diverged
// warp keeps its descriptors in vector registers and moves six of them per MMA into uniform ones,
// which takes 90 cycles and more, whatever the MMA's size (N = 16 to 128 measured alike).  So the
// MMA warp runs its loop undivided, with warp-uniform values throughout, and only the instruction
// itself is predicated on one elected lane: 48 cycles for M = 128, N = 64, K = 16 from shared
// memory (its 6 KB of operands at 128 bytes a cycle), 64 for N = 128 (the tensor rate).

// 1 on one lane of a converged warp, 0 on the others.
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(p));
    return p;
}
// A value equal on all lanes, as one the compiler knows to be uniform.
__device__ __forceinline__ uint32_t uniform(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }

// Reuse of the left operand by the next MMAs: its rows stay in the tensor core's collector from
// the fill to the last use, which leaves the right operand's 2 KB (N = 64) to read per MMA.
enum Collector { kDiscard = 0, kFill = 1, kUse = 2, kLastUse = 3 };

// Operand addresses as the low words of two descriptors with the high word HI, plus constant offsets
// AO, BO (bytes): one 32-bit addition each, where 64-bit descriptors are kept in registers instead.
#define LG_MMA_WARP(kind, qual)                                                                                    \
    asm volatile(                                                                                                  \
        "{\n\t.reg .pred p, q;\n\t.reg .b32 a, b;\n\t.reg .b64 da, db;\n\t"                                         \
        "setp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"                                                       \
        "add.u32 a, %1, %7;\n\tadd.u32 b, %2, %8;\n\tmov.b64 da, {a, %6};\n\tmov.b64 db, {b, %6};\n\t"             \
        "@q tcgen05.mma.cta_group::1.kind::" kind qual " [%0], da, db, %3, p;\n\t}" ::"r"(d_tmem),                 \
        "r"(alo), "r"(blo), "r"(idesc), "r"(accumulate), "r"(elected), "n"(HI), "n"(AO >> 4), "n"(BO >> 4)         \
        : "memory")
template <int COL, uint32_t HI, int AO, int BO>
__device__ __forceinline__ void mma_bf16_warp(uint32_t elected, uint32_t d_tmem, uint32_t alo, uint32_t blo,
                                              uint32_t idesc, uint32_t accumulate) {
    if constexpr (COL == kFill) LG_MMA_WARP("f16", ".collector::a::fill");
    else if constexpr (COL == kUse) LG_MMA_WARP("f16", ".collector::a::use");
    else if constexpr (COL == kLastUse) LG_MMA_WARP("f16", ".collector::a::lastuse");
    else LG_MMA_WARP("f16", "");
}
template <int COL, uint32_t HI, int AO, int BO>
__device__ __forceinline__ void mma_tf32_warp(uint32_t elected, uint32_t d_tmem, uint32_t alo, uint32_t blo,
                                              uint32_t idesc, uint32_t accumulate) {
    if constexpr (COL == kFill) LG_MMA_WARP("tf32", ".collector::a::fill");
    else if constexpr (COL == kUse) LG_MMA_WARP("tf32", ".collector::a::use");
    else if constexpr (COL == kLastUse) LG_MMA_WARP("tf32", ".collector::a::lastuse");
    else LG_MMA_WARP("tf32", "");
}
#undef LG_MMA_WARP

__device__ __forceinline__ void mma_commit_warp(uint32_t elected, uint64_t *mbar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(mbar)),
        "r"(elected)
        : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t *mbar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Wait for phase `parity` of the mbarrier to complete; at most `limit` polls.  Returns false
// on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t *mbar, uint32_t parity, long long limit = kSpinLimit) {
    const uint32_t a = smem_u32(mbar);
    for (long long it = 0; it < limit; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// A wait that does not tell how it ended (for warps that issue MMAs, whose code should not depend on it): the first
// of a CTA that runs out sets *quit (shared memory, zeroed before), which ends the others at their next poll.
__device__ __forceinline__ void mbar_wait_quit(uint64_t *mbar, uint32_t parity, volatile int *quit) {
    long long it = 0;
    for (; it < kSpinLimit; ++it) {
        if (mbar_wait(mbar, parity, 1) || *quit) break;
    }
    if (it == kSpinLimit) *quit = 1;
}

// 32 lanes x 16 consecutive 32-bit columns of TMEM into registers (one warp), which hold the values
// after tmem_wait_ld on them.
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, float (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
          "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
        : "r"(taddr)
        : "memory");
}
// Ties the values to the wait, so that no use of them moves before it.
__device__ __forceinline__ void tmem_touch(float (&v)[16]) {
    asm volatile(""
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]),
                   "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15])
                 :
                 : "memory");
}
template <typename... V>
__device__ __forceinline__ void tmem_wait_ld(V &...v) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    (tmem_touch(v), ...);
}

}  // namespace tc
}  // namespace lg
