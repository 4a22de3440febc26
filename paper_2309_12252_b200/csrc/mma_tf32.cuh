// TF32 tensor-core helpers shared by the kernels whose products run as warp-level m16n8k8 MMAs.
#pragma once
#include "common.cuh"

namespace deer {

// d = a * b + c   (m16n8k8, A row-major 16x8, B 8x8, TF32 inputs, fp32 accumulate)
__device__ __forceinline__ void mma_tf32(float (&d)[4], const unsigned (&a)[4], const unsigned (&b)[2], const float (&c)[4])
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]),
                   "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}

// hi / lo TF32 split by truncation: hi keeps the top 10 mantissa bits, lo the next 10 of the exact
// remainder, so hi*hi + hi*lo + lo*hi carries about 21 mantissa bits of every product.  The tensor
// core reads only the upper 19 bits of a TF32 operand register, so neither half needs masking:
// hi is x itself, lo is x minus its truncation (bit-identical to the masked form on sm_100a).
__device__ __forceinline__ void split_tf32(float x, unsigned &hi, unsigned &lo)
{
    hi = __float_as_uint(x);
    lo = __float_as_uint(x - __uint_as_float(hi & 0xffffe000u));
}

}  // namespace deer
