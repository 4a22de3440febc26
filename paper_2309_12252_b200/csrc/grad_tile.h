// Parameter gradients and dx from the pre-activation gradients in one pass (grad_tile.cu): host-side interface.
#pragma once
#include "common.cuh"

namespace deer {

struct GradTileArgs {
    const float *dGi, *dGh;      // [N,3n] gradients w.r.t. the input-side and hidden-side pre-activations
    const StatusBlock *packed;   // or, where this block's done is set: dGi holds rows [4n] = (r, z, n hidden, n input)
    const float *x, *y, *y0;     // [N,m], [N,n], [B,n]
    const float *W_i;            // [3n,m]
    float *dx;                   // [N,m] or nullptr
    float *slices;               // [CTAs][grad_tile_slice(n, m)]
    int N, T, n, m;
    int expire;                  // test aid: the bounded waits of a CTA's last thread run out (DEER_FLAG_EXPIRE_PRODUCT_WAITS)
    StatusBlock *st;
};

// floats of a slice of the sums: [n + m][4n], then the biases' [4n]
__host__ __device__ constexpr size_t grad_tile_slice(int n, int m) { return (size_t)4 * n * (n + m + 1); }

// Does the launch take these sizes and operands, and has it room for its slices?  `room`: floats of `slices`.
bool grad_tile_suits(const GradTileArgs &a, size_t room);
int launch_grad_tile(const GradTileArgs &a, float *dW_i, float *dW_h, float *db_i, float *db_h, cudaStream_t st);

}  // namespace deer
