// The one-launch Newton kernels of one padded state size: compiled once per size with -DBODY_N=8, 16, ... 64 (build.py).
#include "newton_segment.cuh"
#include "newton_adjoint.cuh"
#include "newton_lane.cuh"
#include "rows_adjoint.cuh"
#include "newton_tile.cuh"

#ifndef BODY_N
#error "BODY_N: state size, a multiple of 8 up to 64"
#endif
#if BODY_N == 64
#include "adjoint_tile.cuh"
#endif

namespace deer {

// v2: rows as 8-byte pairs; exact: products with the update at fp32 level
template <int N> static BodyKernels kernels_of(bool v2, bool exact)
{
    BodyKernels k{};
    if constexpr (N > 8) k.one = v2 ? newton_body_kernel<N, true, true> : newton_body_kernel<N, false, true>;
    k.seg = v2 ? newton_segment_kernel<N, true, true> : newton_segment_kernel<N, false, true>;
    if constexpr (N == 16 || N == 32 || N == 64) {
        // single-TF32 products with the update: the sizes whose solve has always run in reduced precision
        if (v2 && !exact) { k.one = newton_body_kernel<N, true, false>; k.seg = newton_segment_kernel<N, true, false>; }
    }
    constexpr int few = adjoint_ctas<N>(0), many = adjoint_ctas<N>(64);
    k.adj = v2 ? [](int m) -> void (*)(AdjArgs) { return adjoint_ctas<N>(m) == few ? newton_adjoint_kernel<N, true, few> : newton_adjoint_kernel<N, true, many>; }
               : [](int m) -> void (*)(AdjArgs) { return adjoint_ctas<N>(m) == few ? newton_adjoint_kernel<N, false, few> : newton_adjoint_kernel<N, false, many>; };
    if constexpr (N == 32 || N == 64) {
        k.tile = [](int m) -> void (*)(BodyArgs) { return m <= 32 ? newton_tile_kernel<N, 1, true> : newton_tile_kernel<N, 64 / N, false>; };
        k.tile_threads = TileBody<N>::THREADS;
        k.tile_chains = TileBody<N>::GROUPS * TileBody<N>::ROWS;
        k.tile_units = tile_units_kernel<N>;
        k.tile_smem = [](int m) { return TileBody<N>::smem((m + 15) & ~15); };
    }
#if BODY_N == 64
    k.adj_tile = [](int m) -> void (*)(AdjArgs) { return adjoint_tile_kernel; };
    k.adj_tile_smem = [](int m) { return TileAdj::smem((m + 15) & ~15); };
#endif
    k.one_warps = N > 32 ? 8 : 4;
    k.seg_warps = Seg<N, true>::WARPS;
    k.nc_max = Seg<N, true>::NC_MAX;
    k.slot_bytes = Seg<N, true>::SZ * sizeof(float);
    k.one_smem = [](int kx) { return Body<N>::smem(N > 32 ? 8 : 4, kx); };
    k.adj_smem = [](int kx) { return Adj<N>::smem(N > 32 ? 8 : 4, kx); };
    k.seg_fixed = [](int kx) { return Seg<N, true>::fixed(kx); };
    if constexpr (N == 16) { if (v2 && !exact) k.seg_fixed = [](int kx) { return Seg<N, false>::fixed(kx); }; }
    return k;
}

#if BODY_N == 8
template <int N, int M> static LaneKernel lane_of() { return {newton_lane_kernel<N, M>, Lane<N, M>::SMEM, Lane<N, M>::W}; }
template <int N> static LaneKernel lane_m(int m, bool have_u)
{
    if (have_u) return lane_of<N, 0>();
    return m <= 1 ? lane_of<N, 1>() : m <= 2 ? lane_of<N, 2>() : m <= 4 ? lane_of<N, 4>() : lane_of<N, 8>();
}
LaneKernel lane_kernel(int n, int m, bool have_u)
{
    return n <= 1 ? lane_m<1>(m, have_u) : n <= 2 ? lane_m<2>(m, have_u) : n <= 4 ? lane_m<4>(m, have_u) : lane_m<8>(m, have_u);
}
using RowsAdjKernel = void (*)(AdjArgs, RowsAdjOut);
template <int N> static RowsAdjKernel rows_m(int m) { return m == 1 ? rows_adjoint_kernel<N, 1> : m == 2 ? rows_adjoint_kernel<N, 2> : m == 4 ? rows_adjoint_kernel<N, 4> : rows_adjoint_kernel<N, 8>; }
void (*rows_adjoint_of(int n, int m))(AdjArgs, RowsAdjOut) { return n == 1 ? rows_m<1>(m) : n == 2 ? rows_m<2>(m) : n == 4 ? rows_m<4>(m) : rows_m<8>(m); }
int launch_rows_adjoint(const AdjArgs &a, const BodyPlan &p, float *partial_i, float *partial_h, float *dx, cudaStream_t st)
{
    const RowsAdjOut out{partial_i, partial_h, dx};
    DEER_KERNEL("rows_adjoint_kernel", st, rows_adjoint_of(a.n, a.m)<<<(unsigned)p.max_ctas, 128, 0, st>>>(a, out));
    return DEER_OK;
}
#endif

#define BODY_CAT_(a, b) a##b
#define BODY_CAT(a, b) BODY_CAT_(a, b)
BodyKernels BODY_CAT(body_kernels_, BODY_N)(bool v2, bool exact) { return kernels_of<BODY_N>(v2, exact); }

}  // namespace deer
