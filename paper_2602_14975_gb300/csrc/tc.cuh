// Inline-PTX helpers for the 5th-generation tensor cores (tcgen05, sm_100
// and later): shared-memory matrix descriptors, the bf16 MMA with an fp32
// accumulator in tensor memory (TMEM), commits to an mbarrier, TMEM
// allocation and loads.
#pragma once
#include <cstdint>

namespace dmts {

// Shared-memory matrix descriptor of a K-major operand tile with the
// 128-byte swizzle: rows of 128 bytes (64 bf16), 8-row groups 1024 bytes
// apart; `addr` is the tile's (or a 32-byte K-step's) shared address, the
// tile itself 1024-byte aligned.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);        // start address
    d |= (uint64_t)1 << 16;                        // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;              // stride byte offset
    d |= (uint64_t)1 << 46;                        // descriptor version
    d |= (uint64_t)2 << 61;                        // 128-byte swizzle
    return d;
}

// The general form: swizzle 128 or 32 bytes, leading and stride byte offsets.
// Canonical layouts (T = 16-byte units of 8 halves):
//  K-major:  rows of one swizzle span along K, 8-row groups `sbo` apart
//            (`lbo` unused: each MMA's K = 16 lies within a span);
//  MN-major: K rows of one swizzle span (64 or 16 elements) along M / N, 8-row
//            groups `sbo` apart, the next 64 or 16 elements `lbo` further.
__device__ __forceinline__ uint64_t smem_desc_sw(uint32_t addr, uint32_t lbo, uint32_t sbo, int swizzle) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)(swizzle == 128 ? 2 : 6) << 61;
    return d;
}

// Byte offset of the 16-byte chunk j (0, 1) of row r of a 32-byte-swizzled
// tile (rows of 32 bytes, 256-byte aligned): j is XORed with bit 2 of r.
__host__ __device__ __forceinline__ uint32_t swz32(int r, int j) {
    return (uint32_t)r * 32u + ((uint32_t)(j ^ ((r >> 2) & 1)) << 4);
}

// Byte offset, within a 1024-byte-aligned tile in that layout, of the
// 16-byte chunk j (0..7) of row r: the chunk index is XORed with r mod 8.
__host__ __device__ __forceinline__ uint32_t swz128(int r, int j) {
    return (uint32_t)r * 128u + ((uint32_t)(j ^ (r & 7)) << 4);
}

// Instruction descriptor of kind::f16 with bf16 A and B, fp32 D, both
// operands K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// kind::f16 with fp16 A and B, fp32 D; a_mn / b_mn: the operand is MN-major.
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N, int a_mn, int b_mn) {
    return (1u << 4) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

// D[tmem] (+)= A x B^T, M = 128 (cta_group::1), K = 16 (the operand type is the descriptor's).
__device__ __forceinline__ void mma_f16kind(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(accum));
}

// True in one lane of a converged warp. MMAs are issued under it, not under a
// lane-index test: the warp stays uniform, so descriptors are formed in
// uniform registers instead of being moved there for every instruction.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(p));
    return p != 0;
}

// Arrives on the mbarrier once every MMA this thread issued has completed.
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// Warp-collective TMEM allocation of `cols` columns (a power of two >= 32);
// the base address is written to shared memory at `dst`.
__device__ __forceinline__ void tmem_alloc(uint32_t dst, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(cols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols));
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Warp-collective loads of 16 / 8 consecutive fp32 columns of this thread's
// TMEM lane (warp w reads lanes 32(w mod 4) .. + 31; taddr carries the lane
// base in its upper 16 bits), completed before returning.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = __uint_as_float(r[k]);
}

// Issues a load of 8 columns without waiting (tmem_wait_ld completes it).
__device__ __forceinline__ void tmem_ld8_issue(uint32_t taddr, uint32_t *r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

}  // namespace dmts
