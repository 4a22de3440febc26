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
// TF32 MMAs, and good to 2^-22 of its operands where that one is to 2^-20 -- as far as the lo halves are normal f16 numbers, where
// TF32 has the range of fp32: operands need scales.
__device__ __forceinline__ void mma_f16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Powers of two of a cell's f16 operands.  W_h has one, `w`: 2^12, or less where an entry is 4 or more.  The states have one,
// `states` (a constant of the kernel's), and products are accumulated in units of 1 / (w states).  W_i and x have one per
// channel k: the largest weight of the channel comes to 2^`top` and x[k] is multiplied by xf[k], what the accumulators' unit leaves,
// which is 2^-top w states times that weight.  x[k] then counts by what it contributes to a gate, in whatever unit it comes: with top =
// 10 and states = 4 a contribution is good to 2^-22 of itself or 2^-29 absolute, below the 2e-7 of the gates' own arithmetic, up
// to 4,094.  (One power of two for x and one for both matrices held the same cell in other units, x s and W_i / s, to 3e-4 at s =
// 1e-5 and 4e-3 at 1e-6.)
// All threads of the CTA; xf: 64 words of shared memory (m <= 64; m = 0: none of W_i), red: one.  Returns w.
__device__ __forceinline__ float operand_scales(const float *W_h, const float *W_i, int rows, int n, int m, float states, int top, float *xf, unsigned *red)
{
    unsigned *xm = reinterpret_cast<unsigned *>(xf);
    for (int k = threadIdx.x; k < 64; k += blockDim.x) xm[k] = 0u;
    if (threadIdx.x == 0) *red = 0u;
    __syncthreads();
    const auto largest = [](const float *v, int end, int step) {         // (eight loads in flight: the launch waits for this)
        unsigned t = 0u;
        for (int i = threadIdx.x; i < end; i += 8 * step) {
            float w[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) w[j] = i + j * step < end ? v[i + j * step] : 0.0f;
#pragma unroll
            for (int j = 0; j < 8; ++j) t = max(t, __float_as_uint(fabsf(w[j])));
        }
        return t;
    };
    const int threads = blockDim.x, taken = m > 0 ? min(threads / m, 16) * m : 0;    // of W_i a thread to a channel, sixteen at most
    unsigned q = largest(W_h, rows * n, threads);
    const unsigned c = (int)threadIdx.x < taken ? largest(W_i, rows * m, taken) : 0u;
    q = __reduce_max_sync(0xffffffffu, q);
    if ((threadIdx.x & 31) == 0) atomicMax(red, q);
    if (c) atomicMax(xm + (int)threadIdx.x % m, c);
    __syncthreads();
    const auto exponent = [](unsigned bits, int lo, int hi) { return min(max((int)(bits >> 23) - 127, lo), hi); };     // (zero, or beyond any use: the scales stay finite)
    const auto pow2 = [](int e) { return __uint_as_float((unsigned)(127 + e) << 23); };
    const float w = pow2(12 - max(exponent(*red, 0, 60) - 1, 0));
    for (int k = threadIdx.x; k < 64; k += blockDim.x) xf[k] = w * states * pow2(exponent(xm[k], -40, 60) - top);
    __syncthreads();
    return w;
}
// 1 / x of a power of two
__device__ __forceinline__ float pow2_inverse(float x) { return __uint_as_float(0x7f000000u - __float_as_uint(x)); }

}  // namespace deer
