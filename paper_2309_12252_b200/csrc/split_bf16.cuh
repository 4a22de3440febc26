// fp32 operands of tcgen05 products as three bf16 parts.
//
// Three parts of 8 bits, each rounded to nearest, are x exactly (the rest behind two has 7 bits at most); six products (hh, hm, mh,
// mm, hl, lh) leave out 2^-24 of a product at most (2 * 2^-8 * 2^-17), of either sign, where 3 x TF32 with its cut lo part leaves out
// some 2^-20.  (Parts that are cut leave out up to 2^-21, always towards zero: 3e-8 of a sum on average.)  bf16 has the range of fp32,
// so no scale is needed.  The tensor core cuts when it adds to an accumulator: the large products (hh) get accumulators of their
// own, or come last.
#pragma once
#include "tile_umma.cuh"

namespace deer {

// parts of A and B (hi, mid, lo) in the six products, small ones first
__host__ __device__ constexpr int SPLIT_A(int p) { return p == 1 ? 2 : p == 2 || p == 4 ? 1 : 0; }
__host__ __device__ constexpr int SPLIT_B(int p) { return p == 0 ? 2 : p == 2 || p == 3 ? 1 : 0; }

// x = a + b + c; pairs packed.  The first part of a finite x above bf16's largest (3.39e38; a mask may hold the type's lowest value) is
// that largest, not infinity; an infinite x has an infinite second part.
__device__ __forceinline__ void split_bf16(float2 x, unsigned &a, unsigned &b, unsigned &c)
{
    auto pack = [](float2 v) { unsigned d; asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(v.y), "f"(v.x)); return d; };
    auto left = [](float2 v, unsigned d) { return ffma2(make_float2(__uint_as_float(d << 16), __uint_as_float(d & 0xffff0000u)), make_float2(-1.0f, -1.0f), v); };
    asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(a) : "f"(x.y), "f"(x.x));
    const float2 r = left(x, a);
    b = pack(r);
    c = pack(left(r, b));
}

// four values' parts into three operands `part` bytes apart
__device__ __forceinline__ void put_bf16(unsigned char *at, unsigned part, float4 v)
{
    uint2 p[3];
    split_bf16(make_float2(v.x, v.y), p[0].x, p[1].x, p[2].x);
    split_bf16(make_float2(v.z, v.w), p[0].y, p[1].y, p[2].y);
#pragma unroll
    for (int i = 0; i < 3; ++i) *reinterpret_cast<uint2 *>(at + i * part) = p[i];
}

// Instruction descriptor: D fp32, A and B bf16, each K-major or MN-major.
__host__ __device__ constexpr unsigned bf16_idesc(unsigned m, unsigned n, bool a_mn, bool b_mn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (a_mn ? 1u << 15 : 0u) | (b_mn ? 1u << 16 : 0u) | ((n >> 3) << 17) | ((m >> 4) << 24);
}
// XORed to a tile_desc: an MN-major operand over more than one panel, `stride` bytes apart
__host__ __device__ constexpr uint64_t panels_apart(unsigned stride) { return ((uint64_t)(stride >> 4) << 16) ^ (1ull << 16); }

__device__ __forceinline__ void tile_ld16(unsigned taddr, float (&v)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
                   "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
                 : "r"(taddr));
}

}  // namespace deer
