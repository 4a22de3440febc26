// Dense products of any size on tcgen05 at fp32 level (tile_gemm.cu): host-side interface.
#pragma once
#include "newton_body.h"

namespace deer {

struct TileGemmArgs {
    const float *A, *B;      // A(i, k) = A[i * lda + k], or [k * lda + i]; B(j, k) likewise
    size_t lda, ldb;
    int M, N, K;
    const float *bias;       // [N] or nullptr
    float *C;                // [M, N] = A B^T + bias (ldc = N); or, sums: slices [P][N + 1][M] over P parts of K, the last row of
                             // each the sums of A's rows
    // heads: the hidden weights' sums of a multi-head unit (N = n).  A = dG_h [K, H n3]; B = y [K, H n], read a head's stride
    // before (y0 [B, H n] where there is no such row).
    const BodyHead *heads;
    const float *y0;
    int T, n, n3;
    int expire;              // test aid: the bounded waits of a CTA's last thread run out (DEER_FLAG_EXPIRE_PRODUCT_WAITS)
    StatusBlock *st;
    int chunks;              // (set by the launch)
};

enum class TileGemm { MAP, MAP_T, SUMS, SUMS_HEADS };    // B rows [N][K]; B rows [K][N]; A and B rows [K][.], slices; see `heads`
int launch_tile_gemm(TileGemm form, const TileGemmArgs &a, int P, cudaStream_t st);
// Slices for a SUMS launch that fills the GPU, at most `room`.
int tile_gemm_slices(int M, int N, int K, int room);

}  // namespace deer
