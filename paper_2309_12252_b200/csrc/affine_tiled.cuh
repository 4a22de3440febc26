// Dense affine map of any size on tensor cores: out[e][c] = bias[c] + sum_k W(c,k) in[e][k], W(c,k) = W[c*K + k] or, WT,
// W[k*NOUT + c].  The stacked input projections of a multi-head unit ([B*T, m] x [m, 3nH]) and their gradient
// ([B*T, 3nH] x [3nH, m]): affine_mma_kernel keeps the whole weight matrix in shared memory, which these do not fit.
//
// CTA tile 128 x 64, K in chunks of 32 through a ring of three cp.async stages; warp tile 32 x 32 of m16n8k8 TF32 MMAs, issued
// three times on hi/lo splits (fp32-level accuracy).  Bound by the MMA issue rate: 24 MMAs (about 195 cycles of a sub-partition)
// against about 50 other instructions per 8 k and warp.  The contraction index of a K step is renamed (slots t, t + 4 hold
// 2t, 2t + 1), so that a lane's operands are adjacent pairs; row strides are 8 (mod 32) words: conflict-free.
#pragma once
#include "mma_tf32.cuh"
#include "scan_onepass.cuh"

namespace deer {

struct AffineTile {
    static constexpr int MT = 128, NT = 64, KT = 32, STAGES = 3, THREADS = 256;
    static constexpr int AS = KT + 8;                    // row stride of the A tile and of the B tile [out][in]
    static constexpr int BS = NT + 4;                    // row stride of the B tile [in][out]
    static constexpr int BTILE = NT * AS > KT * BS ? NT * AS : KT * BS;
    static constexpr int STAGE = MT * AS + BTILE;
    static constexpr size_t SMEM = sizeof(float) * STAGES * STAGE;
};

template <bool WT>
__global__ void __launch_bounds__(256, 2) affine_tiled_kernel(const float *__restrict__ in, const float *__restrict__ W,
                                                              const float *__restrict__ bias, float *__restrict__ out, size_t N,
                                                              int K, int NOUT, int vec)
{
    using C = AffineTile;
    extern __shared__ __align__(16) float sma[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const int ct = (NOUT + C::NT - 1) / C::NT;           // consecutive CTAs share their rows of `in`
    const size_t r0 = (size_t)(blockIdx.x / ct) * C::MT;
    const int c0 = (int)(blockIdx.x % ct) * C::NT;
    const int wr = (warp >> 1) * 32, wc = (warp & 1) * 32;
    const int nk = (K + C::KT - 1) / C::KT;

    // one operand tile: `rows` rows of `width` floats from src (pitch ld), zero where row >= rmax or column >= cmax
    auto tile = [&](float *dst, int stride, int rows, int width, const float *src, size_t ld, size_t row0, size_t rmax, int col0, int cmax) {
        if (vec) {
            const int q = width >> 2;
            for (int i = tid; i < rows * q; i += C::THREADS) {
                const int r = i / q, c = 4 * (i - r * q);
                float *d = dst + r * stride + c;
                if (row0 + r < rmax && col0 + c < cmax) cp_async16(d, src + (row0 + r) * ld + col0 + c);
                else *reinterpret_cast<float4 *>(d) = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        } else {
            for (int i = tid; i < rows * width; i += C::THREADS) {
                const int r = i / width, c = i - r * width;
                dst[r * stride + c] = row0 + r < rmax && col0 + c < cmax ? __ldg(src + (row0 + r) * ld + col0 + c) : 0.0f;
            }
        }
    };
    auto issue = [&](int k) {
        if (k < nk) {
            float *sA = sma + (k % C::STAGES) * C::STAGE, *sB = sA + C::MT * C::AS;
            tile(sA, C::AS, C::MT, C::KT, in, (size_t)K, r0, N, k * C::KT, K);
            if constexpr (WT) tile(sB, C::BS, C::KT, C::NT, W, (size_t)NOUT, (size_t)k * C::KT, (size_t)K, c0, NOUT);
            else tile(sB, C::AS, C::NT, C::KT, W, (size_t)K, (size_t)c0, (size_t)NOUT, k * C::KT, K);
        }
        cp_async_commit();
    };
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
    issue(0);
    issue(1);
#pragma unroll 1
    for (int k = 0; k < nk; ++k) {
        static_assert(C::STAGES == 3, "the wait below leaves one group in flight");
        cp_async_wait_1();
        __syncthreads();                                 // chunk k landed for every thread; the stage of chunk k - 1 is free
        issue(k + 2);
        const float *sA = sma + (k % C::STAGES) * C::STAGE + (wr + g) * C::AS + 2 * t;
        const float *sB = sma + (k % C::STAGES) * C::STAGE + C::MT * C::AS;
#pragma unroll
        for (int k0 = 0; k0 < C::KT; k0 += 8) {
            unsigned ah[2][4], al[2][4];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float2 x0 = *reinterpret_cast<const float2 *>(sA + 16 * i * C::AS + k0);
                const float2 x1 = *reinterpret_cast<const float2 *>(sA + (16 * i + 8) * C::AS + k0);
                split_tf32(x0.x, ah[i][0], al[i][0]);
                split_tf32(x1.x, ah[i][1], al[i][1]);
                split_tf32(x0.y, ah[i][2], al[i][2]);
                split_tf32(x1.y, ah[i][3], al[i][3]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float b0, b1;
                if constexpr (WT) {
                    const float *q = sB + (k0 + 2 * t) * C::BS + wc + 8 * j + g;
                    b0 = q[0]; b1 = q[C::BS];
                } else {
                    const float2 w = *reinterpret_cast<const float2 *>(sB + (wc + 8 * j + g) * C::AS + k0 + 2 * t);
                    b0 = w.x; b1 = w.y;
                }
                unsigned bh[2], bl[2];
                split_tf32(b0, bh[0], bl[0]);
                split_tf32(b1, bh[1], bl[1]);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    mma_tf32(acc[i][j], al[i], bh, acc[i][j]);
                    mma_tf32(acc[i][j], ah[i], bl, acc[i][j]);
                    mma_tf32(acc[i][j], ah[i], bh, acc[i][j]);
                }
            }
        }
    }
    cp_async_wait_0();
    const bool pair = (NOUT & 1) == 0 && ((uintptr_t)out & 7) == 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int c = c0 + wc + 8 * j + 2 * t;
        const float b0 = bias && c < NOUT ? bias[c] : 0.0f, b1 = bias && c + 1 < NOUT ? bias[c + 1] : 0.0f;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const size_t r = r0 + wr + 16 * i + 8 * h + g;
                if (r >= N) continue;
                float *o = out + r * NOUT + c;
                const float v0 = acc[i][j][2 * h] + b0, v1 = acc[i][j][2 * h + 1] + b1;
                if (pair) { if (c < NOUT) *reinterpret_cast<float2 *>(o) = make_float2(v0, v1); }
                else { if (c < NOUT) o[0] = v0; if (c + 1 < NOUT) o[1] = v1; }
            }
    }
}

}  // namespace deer
