// tcgen05 building blocks of the kernels whose chains are the 128 rows of a tensor-core tile: f16 operands in shared memory
// (K-major, SWIZZLE_128B panels of 64 columns), fp32 accumulators in tensor memory.
#pragma once
#include "scan_onepass.cuh"
#include "split_f16.cuh"

namespace deer {

// Byte offset of 16-bit element (row, k) in an operand of `rows` rows: panels of 64 columns, 128 bytes a row, the 16-byte
// pieces of a row XORed with row % 8.
__device__ __forceinline__ unsigned panel_off(unsigned rows, unsigned row, unsigned k)
{
    return (k >> 6) * (rows * 128u) + row * 128u + ((((k & 63u) >> 3) ^ (row & 7u)) << 4) + ((k & 7u) << 1);
}
// What the K step that starts at column k (a multiple of 16) adds to a descriptor
__device__ __forceinline__ uint64_t panel_k(unsigned rows, unsigned k) { return ((k >> 6) * (rows * 128u) + (k & 63u) * 2u) >> 4; }

// Shared-memory matrix descriptor: start address, stride between groups of 8 rows (1024 bytes), version 1, SWIZZLE_128B.
// (K steps and row blocks add their byte offset >> 4 to it.)
__device__ __forceinline__ uint64_t tile_desc(unsigned saddr)
{
    return (uint64_t)((saddr >> 4) & 0x3FFF) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// The same for operands of 32 columns: 64 bytes a row, SWIZZLE_64B (pieces XORed with row / 2 % 4, groups of 512 bytes).
__device__ __forceinline__ unsigned narrow_off(unsigned row, unsigned k)
{
    return row * 64u + (((k >> 3) ^ ((row >> 1) & 3u)) << 4) + ((k & 7u) << 1);
}
__device__ __forceinline__ uint64_t narrow_desc(unsigned saddr)
{
    return (uint64_t)((saddr >> 4) & 0x3FFF) | (1ull << 16) | ((uint64_t)(512 >> 4) << 32) | (1ull << 46) | (4ull << 61);
}

// Instruction descriptor: D fp32, A and B f16, both K-major, M = 128.
__host__ __device__ constexpr unsigned tile_idesc(unsigned n) { return (1u << 4) | ((n >> 3) << 17) | ((128u >> 4) << 24); }

// One lane of a converged warp: issued under a warp-uniform branch, the descriptors stay in uniform registers.
__device__ __forceinline__ bool tile_elect()
{
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(ok));
    return ok != 0;
}

__device__ __forceinline__ void tile_mma(unsigned tmem_d, uint64_t a, uint64_t b, unsigned idesc, unsigned accumulate)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p; \n\t"
        "}\n"
        :
        : "r"(tmem_d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

// A from tensor memory (row = lane, two f16 per 32-bit column); B K-major, or MN-major with tile_idesc's bit 16
__device__ __forceinline__ void tile_mma_ta(unsigned tmem_d, unsigned tmem_a, uint64_t b, unsigned idesc, unsigned accumulate)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p; \n\t"
        "}\n"
        :
        : "r"(tmem_d), "r"(tmem_a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
constexpr unsigned TILE_B_MN = 1u << 16;

__device__ __forceinline__ void tile_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// four accumulator columns of this thread's row
__device__ __forceinline__ void tile_ld4(unsigned taddr, float2 (&v)[2])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[1].x), "=f"(v[1].y)
                 : "r"(taddr));
}
__device__ __forceinline__ void tile_st2(unsigned taddr, unsigned a, unsigned b)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(taddr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void tile_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tile_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tile_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tile_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Bounded wait for a phase of an mbarrier; false when it gives up.
constexpr unsigned TILE_SPIN_LIMIT = 1u << 24;
__device__ __forceinline__ bool tile_wait(uint64_t *bar, unsigned phase)
{
    const unsigned addr = smem_u32(bar);
    for (unsigned spins = 0; spins < TILE_SPIN_LIMIT; ++spins) {
        unsigned ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
                     : "=r"(ok)
                     : "r"(addr), "r"(phase)
                     : "memory");
        if (ok) return true;
    }
    return false;
}

}  // namespace deer
