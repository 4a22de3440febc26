// fp32 values as hi + lo f16 halves, and the warp-level MMA on them.
#pragma once
#include "common.cuh"
#include <cuda_fp16.h>

namespace deer {

// hi and lo halves of a pair as packed f16: x = hi + lo to 2^-23 of x, or 2^-25 where lo is subnormal (|x| below 2^-2; values up
// to 65504)
__device__ __forceinline__ void split_f16(float2 x, unsigned &hi, unsigned &lo)
{
    const __half2 h = __float22half2_rn(x);
    const __half2 l = __float22half2_rn(ffma2(__half22float2(h), make_float2(-1.0f, -1.0f), x));
    hi = *reinterpret_cast<const unsigned *>(&h);
    lo = *reinterpret_cast<const unsigned *>(&l);
}
__device__ __forceinline__ unsigned pack_f16(float2 x)
{
    const __half2 h = __float22half2_rn(x);
    return *reinterpret_cast<const unsigned *>(&h);
}

// d += a * b   (m16n8k16, A row-major 16x16, B 16x8, f16 inputs, fp32 accumulate).  It takes the tensor pipe as long as a TF32 MMA of
// eight columns (8.04 and 8.05 cycles a sub-partition), so a product in three of these on hi + lo f16 halves is half of one in three
// TF32 MMAs, and good to 2^-23 of its operands where that one is to 2^-20.
__device__ __forceinline__ void mma_f16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The power of two that brings the largest of `count` weights (and of a second array) to [2^9, 2^10): with it the lo halves
// of all but the very smallest are normal f16 numbers.  All threads of the CTA; red: one word.
__device__ __forceinline__ float tile_weight_scale(const float *w0, int n0, const float *w1, int n1, unsigned *red)
{
    unsigned top = 0u;
    for (int i = threadIdx.x; i < n0; i += blockDim.x) top = max(top, __float_as_uint(fabsf(w0[i])));
    for (int i = threadIdx.x; i < n1; i += blockDim.x) top = max(top, __float_as_uint(fabsf(w1[i])));
    if (threadIdx.x == 0) *red = 0u;
    __syncthreads();
    top = __reduce_max_sync(0xffffffffu, top);
    if ((threadIdx.x & 31) == 0) atomicMax(red, top);
    __syncthreads();
    const int e = min(max((int)(*red >> 23), 40), 220);          // (zero, or beyond any use: the scale stays finite)
    return __uint_as_float((unsigned)(127 + 9 - (e - 127)) << 23);
}

}  // namespace deer
