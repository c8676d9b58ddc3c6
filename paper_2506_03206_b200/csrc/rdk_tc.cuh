// Tensor-core plumbing shared by the tcgen05 kernels: bounded mbarrier waits, operand descriptors, tensor-memory
// loads, tensor maps.
#pragma once

#include <cuda.h>

#include "rdk_common.cuh"

namespace rdk {

constexpr unsigned kTcSpin = 1u << 21;

__device__ __forceinline__ uint32_t s32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Bounded wait on an mbarrier phase; false (and *abort set) when the limit is reached or another
// role has already given up.
// Called by all lanes of a warp; the answer is the same in every lane.
__device__ __forceinline__ bool tc_wait(unsigned long long* bar, uint32_t parity, volatile int* abort) {
    bool ok = false;
    for (unsigned spins = 0; spins < kTcSpin; ++spins) {
        uint32_t done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done) : "r"(s32(bar)), "r"(parity) : "memory");
        if (done) { ok = true; break; }
        if (*abort) break;
    }
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) *abort = 1;
    return ok;
}

// true in one lane of a converged warp, in a form the compiler knows to be uniform
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(p));
    return p != 0;
}

// shared-memory matrix descriptor: K-major operand, rows of 128 bytes, 128-byte swizzle, groups of
// 8 rows 1024 bytes apart
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);         // start address
    d |= (uint64_t)1 << 16;                          // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;                // stride byte offset
    d |= (uint64_t)1 << 46;                          // descriptor version of this architecture
    d |= (uint64_t)2 << 61;                          // 128-byte swizzle
    return d;
}

// D += A B for one 64-wide K block of K-major operands: four instructions of 16, 32 bytes apart in either operand.  One
// thread issues everything, so the descriptors come prepared and an instruction costs it a few adds: built anew for every
// instruction they took 195 to 250 cycles each, whatever the tile, against 128 for the largest.
#define RDK_MMA_KBLOCK(GROUP)                                                                                        \
    asm volatile("{\n .reg .pred p, q;\n .reg .b64 a, b;\n setp.ne.b32 p, %4, 0;\n setp.eq.b32 q, 0, 0;\n"           \
                 " tcgen05.mma.cta_group::" GROUP ".kind::f16 [%0], %1, %2, %3, p;\n"                                \
                 " add.u64 a, %1, 2;\n add.u64 b, %2, 2;\n tcgen05.mma.cta_group::" GROUP ".kind::f16 [%0], a, b, %3, q;\n" \
                 " add.u64 a, %1, 4;\n add.u64 b, %2, 4;\n tcgen05.mma.cta_group::" GROUP ".kind::f16 [%0], a, b, %3, q;\n" \
                 " add.u64 a, %1, 6;\n add.u64 b, %2, 6;\n tcgen05.mma.cta_group::" GROUP ".kind::f16 [%0], a, b, %3, q;\n}" \
                 ::"r"(d), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate ? 1u : 0u) : "memory")
template <int CTA_GROUP>
__device__ __forceinline__ void mma_kblock(uint32_t d, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, bool accumulate) {
    if (CTA_GROUP == 2) RDK_MMA_KBLOCK("2"); else RDK_MMA_KBLOCK("1");
}

// 32 consecutive columns of this warp's 32 TMEM lanes: v[c] is column c of the lane's row
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr) : "memory");
}
// The loads before it have landed; the registers go through it so that no use of them is moved up.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&v)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 32; ++q) asm volatile("" : "+r"(v[q]));
}

// A [outer, inner] matrix of bf16 with rows of pitch_elems elements, read or written in boxes of box_outer rows of
// box_inner elements, 128-byte swizzle; what lies outside reads as zero and is not written.
int make_map(CUtensorMap* map, const void* base, uint64_t inner, uint64_t outer, uint64_t pitch_elems, uint32_t box_inner, uint32_t box_outer);

}  // namespace rdk
