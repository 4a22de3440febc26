// One Newton body as one launch for n = 32 and 64: the solve of newton_body.cuh (chains with a burn-in, boundaries verified;
// see there) with 128 chains in lockstep as the rows of a tcgen05 tile.
//
// Per step of a CTA, [128, .] x [., 3n] products by tcgen05.mma.kind::f16 from one thread, accumulators in tensor memory:
//     x_t W_i^T and y_{t-1} W_h^T   operands as hi + lo f16 halves, three products (good to 2^-22 of the operands and, of small
//                                   ones, to 2^-29 of a state and 2^-27 or better of what x contributes to a gate (tile_usual):
//                                   below the 2e-7 that the gates' tanh is good to)
//     d_{t-1} W_h^T                 one product (the solve's accuracy is that of its boundaries, see body_verdict)
// Operands carry powers of two (operand_scales; OP_SCALE, D_SCALE) that keep the hi halves, and the lo halves of all but small
// operands, among the normal f16 numbers and leave in the exponent arithmetic of the epilogue.  A value beyond f16's range turns the body's error into a NaN: the body
// does not count and the evaluation goes on with the other kernels (BODY_FALL_BACK).
// A row is owned by n/16 threads of one lane, 16 columns each (the warps of a warpgroup see their own 32 tensor-memory lanes):
// gates, coefficients, the update and the new iterate are elementwise in registers.  Loading is another mapping -- a row's
// lanes side by side, full lines per request, a step ahead in registers -- and hands the rows over as f16 operands and, in
// fp32, through `sY`.
//
// What bounds it: the latency of a step's serial phases with 16 warps per SM (128 registers a thread).  n = m = 32, B = 16,
// T = 5.6e4: issue slots 49 % used, special functions 29 %, FMA 34 %, ALU 32 %, tensor 15 %, DRAM 27 %; per instruction issued 1.4
// warps wait for a fixed latency, 1.4 for a load (tensor memory, global), 1.3 at a barrier.  n = 64 (one tile per CTA): issue
// 38 %, 2.8 at a barrier.  mma.sync spent 2,700 of a warp's 5,400 cycles per 16 rows in the tensor pipe alone.
#pragma once
#include "newton_body.cuh"
#include "tile_umma.cuh"

namespace deer {

// a row's chain: position index and time step at step 0, end of its positions (0: idle row), sequence
// (position indices fit: 2^31 of them are 256 GB of states)
struct __align__(16) TileRow { int e, ts, te, b; };

template <int N> struct TileBody {
    static constexpr int GROUPS = N == 32 ? 2 : 1;       // tiles of a CTA, each with its own threads: one's tensor-core products run
                                                         // beside the other's epilogue
    static constexpr int GT = 8 * N, THREADS = GROUPS * GT, ROWS = 128;
    static constexpr int LPR = N / 4;                    // lanes that load a row
    static constexpr int YS = N + 4;                     // stride of sY
    static constexpr unsigned PANEL = 128 * 128;         // bytes of an A panel
    static constexpr unsigned HP = 2 * N / 64;           // panels of the y operand (hi | lo)
    static constexpr unsigned DP = 128 * 2 * N;          // bytes of the d operand
    static constexpr unsigned WROWS = 3 * N;
    static constexpr unsigned TMEM = 512;                // columns of a group: q r z un (n each), d W_h^T (3n)
    __host__ __device__ static constexpr unsigned xp(int kx) { return (2 * kx + 63) / 64; }
    // The y and x operands are double-buffered where they fit: the next step's are put away while this step's products run.
    __host__ __device__ static constexpr bool twice(int kx) { return kx <= 32; }
    __host__ __device__ static constexpr unsigned operands(int kx) { return (twice(kx) ? 2 : 1) * PANEL * (HP + xp(kx)) + DP; }
    static constexpr size_t smem(int kx)
    {
        return 1024 + GROUPS * (size_t)operands(kx) + (size_t)WROWS * 128 * (HP + xp(kx)) +
               sizeof(float) * (GROUPS * ROWS * YS + 4 * N) + GROUPS * sizeof(TileRow) * ROWS;
    }
};

// Scales of the states (up to 4,094) and of the update.
constexpr float TILE_OP_SCALE = 16.0f, TILE_D_SCALE = 1024.0f;

// Inputs have the states' scale where every channel's largest weight is of a usual size, 2^-6 to 4: what x contributes to a gate
// is then held to 2^-27 absolute, up to 64 or more.  Channels in other units are brought to theirs by tile_units_kernel, once per
// evaluation, and the kernel is launched again (`units`): contributions are held to 2^-31, up to 1,023.  A factor per channel in
// the loop, where the weights need none, costs the two-tile form its schedule at 128 registers (n = m = 32, B = 16, T = 1e5:
// 1262 -> 1345 us) and n = 64 a hundredth.
constexpr int TILE_TOP = 10;
__device__ __forceinline__ bool tile_usual(const float *xf, float w, int m, int k)
{
    if (k >= m) return true;
    const int e = (int)(__float_as_uint(xf[k]) >> 23) - (int)(__float_as_uint(w * TILE_OP_SCALE) >> 23) + TILE_TOP;
    return (e >= -6 && e <= 1) || e == -40;                              // (-40: no weights)
}

// x in the units that the tile kernel's operands have (W_i' comes with its own inverse factors)
template <int N> __global__ void __launch_bounds__(256) tile_units_kernel(const float *x, float *xs, size_t count, int m, const float *W_h, const float *W_i)
{
    __shared__ __align__(16) float s_xf[64];
    __shared__ unsigned s_top;
    operand_scales(W_h, W_i, 3 * N, N, m, TILE_OP_SCALE, TILE_TOP, s_xf, &s_top);
    const size_t step = (size_t)gridDim.x * blockDim.x;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += step) xs[i] = x[i] * (s_xf[i % (size_t)m] * (1.0f / TILE_OP_SCALE));
}

template <int N, int XJ, bool TWICE>
__global__ void __launch_bounds__(TileBody<N>::THREADS, 1) newton_tile_kernel(BodyArgs a)
{
    using C = TileBody<N>;
    constexpr unsigned WR = C::WROWS;
    constexpr float LOG2E = 1.4426950408889634f;
    StatusBlock *st = a.st;
    if (*(volatile int *)&st->done) return;

    extern __shared__ __align__(16) unsigned char smem_tile[];
    __shared__ __align__(8) uint64_t s_bars[C::GROUPS];
    __shared__ unsigned s_tmem, s_top;
    __shared__ __align__(16) float s_xf[64];
    __shared__ int s_aborts[C::GROUPS], s_sides[C::GROUPS][2];
    unsigned char *sm = (unsigned char *)(((uintptr_t)smem_tile + 1023) & ~(uintptr_t)1023);
    const int m = a.m, kx = (m + 15) & ~15;
    const int all = threadIdx.x, grp = all / C::GT, tid = all % C::GT, lane = tid & 31, warp = tid >> 5;       // (tid, warp: of the group)
    const unsigned buf = C::PANEL * (C::HP + C::xp(kx));                 // one buffer: y operand, x operand
    unsigned char *sWh = sm, *sWi = sWh + WR * 128 * C::HP;
    unsigned char *sH = sWi + WR * 128 * C::xp(kx) + grp * C::operands(kx), *sX = sH + C::PANEL * C::HP, *sD = sH + (TWICE ? 2 : 1) * buf;
    float *sb = reinterpret_cast<float *>(sWi + WR * 128 * C::xp(kx) + C::GROUPS * C::operands(kx));
    float *sY = sb + 4 * N + grp * C::ROWS * C::YS;
    TileRow *rows = reinterpret_cast<TileRow *>(sb + 4 * N + C::GROUPS * C::ROWS * C::YS) + grp * C::ROWS;
    uint64_t &s_bar = s_bars[grp];
    int &s_abort = s_aborts[grp];
    int *s_side = s_sides[grp];
    auto group_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "r"(C::GT) : "memory"); };
    const long long tile = (long long)grp * gridDim.x + blockIdx.x;      // (few tiles: each on an SM of its own)
    const int L = a.L, T = a.T, nchain = (T + L - 1) / L;
    const long long total = (long long)a.B * nchain;

    // ---- weights, biases, geometry, tensor memory
    const float wscale = operand_scales(a.h0.W_h, a.h0.W_i, 3 * N, N, m, TILE_OP_SCALE, TILE_TOP, s_xf, &s_top);
    const float kS = 1.0f / (wscale * TILE_OP_SCALE), kD = 1.0f / (wscale * TILE_D_SCALE);
    if (!a.units) {
        if (!__syncthreads_and(tile_usual(s_xf, wscale, m, all))) {      // the inputs' units are for tile_units_kernel
            if (all == 0 && blockIdx.x == 0) {
                st->done = BODY_UNITS;
                if (HostResult *h = st->host) { h->burn = st->burn; post_done(h, BODY_UNITS); }
            }
            return;
        }
        if (all < 64) s_xf[all] = TILE_OP_SCALE;
        __syncthreads();
    }
    for (int i = all; i < (int)WR * (N / 2); i += C::THREADS) {          // rows of W_h in the order n, r, z
        const int k = 2 * (i % (N / 2)), r = i / (N / 2), gate = r < N ? 2 : r / N - 1;
        const float2 v = *reinterpret_cast<const float2 *>(a.h0.W_h + (size_t)(gate * N + r % N) * N + k);
        unsigned hi, lo;
        split_f16(make_float2(v.x * wscale, v.y * wscale), hi, lo);
        *reinterpret_cast<unsigned *>(sWh + panel_off(WR, r, k)) = hi;
        *reinterpret_cast<unsigned *>(sWh + panel_off(WR, r, N + k)) = lo;
    }
    for (int i = all; i < (int)WR * (kx / 2); i += C::THREADS) {         // rows of W_i in the order r, z, n
        const int k = 2 * (i % (kx / 2)), r = i / (kx / 2);
        const float *w = a.h0.W_i + (size_t)r * m + k;
        unsigned hi, lo;
        const float unit = wscale * TILE_OP_SCALE;
        split_f16(make_float2(k < m ? w[0] * (unit * pow2_inverse(s_xf[k])) : 0.0f, k + 1 < m ? w[1] * (unit * pow2_inverse(s_xf[k + 1])) : 0.0f), hi, lo);
        *reinterpret_cast<unsigned *>(sWi + panel_off(WR, r, k)) = hi;
        *reinterpret_cast<unsigned *>(sWi + panel_off(WR, r, kx + k)) = lo;
    }
    for (int i = all; i < N; i += C::THREADS) {
        sb[i] = -LOG2E * (a.h0.b_h[i] + a.h0.b_i[i]);
        sb[N + i] = -LOG2E * (a.h0.b_h[N + i] + a.h0.b_i[N + i]);
        sb[2 * N + i] = a.h0.b_h[2 * N + i];
        sb[3 * N + i] = a.h0.b_i[2 * N + i];
    }
    const int iters = *(volatile int *)&st->iters, burn = *(volatile int *)&st->burn;
    if (tid < C::ROWS) {
        const long long gid = tile * C::ROWS + tid;
        TileRow r{0, 0, 0, 0};
        if (gid < total) {
            const long long b = gid / nchain;
            const int c = (int)(gid - b * nchain);
            r.ts = c * L - burn;
            r.te = min(T, (c + 1) * L);
            r.e = (int)(b * T + r.ts);
            r.b = (int)b;
        }
        rows[tid] = r;
    }
    if (tid == 0) { mbar_init(&s_bar, 1); s_abort = 0; s_side[0] = s_side[1] = 0; }
    if (all < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(C::TMEM) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tile_fence_before();
    __syncthreads();
    tile_fence_after();
    const unsigned tmem = s_tmem + (unsigned)grp * 7 * N;

    const float *ycur = a.buf[iters & 1];
    float *ynew = a.buf[(iters + 1) & 1];
    const bool zero = iters == 0 && !a.warm;             // the guess is zero: nothing of it is read
    const int xv = (m & 3) == 0 && ((uintptr_t)a.x & 15) == 0 ? 4 : (m & 1) == 0 && ((uintptr_t)a.x & 7) == 0 ? 2 : 1;

    // ---- loader mapping: rows lr + 32 i, columns 4 lc .. 4 lc + 3 (of x also 4 lc + N ..)
    const int lr = tid / C::LPR, lc = tid % C::LPR;
    // (Loads are unconditional, from addresses that exist, and what is not wanted is zeroed when it is put away: a load under a
    // branch would be waited for where the branch joins.)
    float4 yv[4], xr[4][XJ];
    unsigned y_in = 0u, x_in = 0u;                       // rows (bit i) whose value counts
    // the iterate at every row's step `sy` (y0 just before the sequence), x at step `sx`
    auto load_y = [&](int sy) {
        y_in = 0u;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const TileRow r = rows[lr + 32 * i];
            const int t = r.ts + sy;
            const bool in = t >= 0 && t < r.te && !zero, first = t == -1 && r.te > 0;
            const float *p = (in ? ycur : a.y0) + (size_t)(unsigned)(in ? r.e + sy : r.b) * N;
            y_in |= (in || first ? 1u : 0u) << i;
            yv[i] = __ldcg(reinterpret_cast<const float4 *>(p) + lc);
        }
    };
    auto load_x = [&](int sx) {
        x_in = 0u;
        const float *p[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const TileRow r = rows[lr + 32 * i];
            const int t = r.ts + sx;
            const bool in = t >= 0 && t < r.te;
            x_in |= (in ? 1u : 0u) << i;
            p[i] = a.x + (size_t)(unsigned)(in ? r.e + sx : 0) * m;
        }
#pragma unroll
        for (int j = 0; j < XJ; ++j) {
            const int c = 4 * lc + N * j;
            if (xv == 4) {
                const int cc = min(c, m - 4);
#pragma unroll
                for (int i = 0; i < 4; ++i) xr[i][j] = __ldg(reinterpret_cast<const float4 *>(p[i] + cc));
            } else if (xv == 2) {
                const int ca = min(c, m - 2), cb = min(c + 2, m - 2);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 u = __ldg(reinterpret_cast<const float2 *>(p[i] + ca)), v = __ldg(reinterpret_cast<const float2 *>(p[i] + cb));
                    xr[i][j] = make_float4(u.x, u.y, v.x, v.y);
                }
            } else {
                const int c1 = min(c, m - 1), c2 = min(c + 1, m - 1), c3 = min(c + 2, m - 1), c4 = min(c + 3, m - 1);
#pragma unroll
                for (int i = 0; i < 4; ++i) xr[i][j] = make_float4(__ldg(p[i] + c1), __ldg(p[i] + c2), __ldg(p[i] + c3), __ldg(p[i] + c4));
            }
        }
    };
    auto put = [&](unsigned char *panel, int row, int k, int klo, float4 v) {
        const float2 sc = make_float2(TILE_OP_SCALE, TILE_OP_SCALE);
        uint2 hi, lo;
        split_f16(fmul2(make_float2(v.x, v.y), sc), hi.x, lo.x);
        split_f16(fmul2(make_float2(v.z, v.w), sc), hi.y, lo.y);
        *reinterpret_cast<uint2 *>(panel + panel_off(128, row, k)) = hi;
        *reinterpret_cast<uint2 *>(panel + panel_off(128, row, klo + k)) = lo;
    };
    auto wanted = [](bool in, float4 v) { return in ? v : make_float4(0.f, 0.f, 0.f, 0.f); };
    const bool whole = (m & 3) == 0;                     // a lane's four columns of x are all there or none
    auto put_x = [&](unsigned char *panel) {
#pragma unroll
        for (int j = 0; j < XJ; ++j) {
            const int c = 4 * lc + N * j;
            if (c >= kx) continue;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float4 v = wanted((x_in >> i) & 1u && c < m, xr[i][j]);
                if (!whole) { v.y = c + 1 < m ? v.y : 0.f; v.z = c + 2 < m ? v.z : 0.f; v.w = c + 3 < m ? v.w : 0.f; }
                put(panel, lr + 32 * i, c, kx, v);
            }
        }
    };
    auto put_h = [&](unsigned char *panel) {
#pragma unroll
        for (int i = 0; i < 4; ++i) put(panel, lr + 32 * i, 4 * lc, N, wanted((y_in >> i) & 1u, yv[i]));
    };
    auto put_y = [&]() {
#pragma unroll
        for (int i = 0; i < 4; ++i) *reinterpret_cast<float4 *>(sY + (lr + 32 * i) * C::YS + 4 * lc) = wanted((y_in >> i) & 1u, yv[i]);
    };
    auto d_off = [&](int row, int k) { return N == 32 ? narrow_off(row, k) : panel_off(128, row, k); };

    // ---- owner mapping: row and 16 columns of this thread
    const int row = (warp & 3) * 32 + lane, c0 = (warp >> 2) * 16;
    const TileRow own = rows[row];
    const long long gid = tile * C::ROWS + row;
    const unsigned tacc = tmem + ((unsigned)(32 * (warp & 3)) << 16) + c0;
    const int chain = (int)(gid % nchain);
    const bool has_next = own.te > 0 && chain + 1 < nchain, has_prev = own.te > 0 && chain > 0;
    float2 d[8], hv[8];
    const int s0 = nchain == 1 ? burn : 0, s_end = tile * C::ROWS < total ? burn + min(L, T) : s0;      // (a tile without rows: no steps)

    load_y(s0 - 1);
    load_x(s0);
    put_y();
    put_h(sH);
    put_x(sX);
    group_sync();
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        hv[j] = *reinterpret_cast<const float2 *>(sY + row * C::YS + c0 + 2 * j);
        d[j] = make_float2(0.f, 0.f);
    }
    load_y(s0);
    load_x(s0 + 1);
#pragma unroll
    for (int q = 0; q < 2; ++q) *reinterpret_cast<uint4 *>(sD + d_off(row, c0 + 8 * q)) = make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async();
    tile_fence_before();
    group_sync();

    // warp-uniform copies for the issuing warp
    const int uwarp = __shfl_sync(0xffffffffu, warp, 0);
    const unsigned utmem = __shfl_sync(0xffffffffu, tmem, 0), usH = __shfl_sync(0xffffffffu, smem_u32(sH), 0);
    const uint64_t dH0 = tile_desc(usH), dX0 = tile_desc(usH + C::PANEL * C::HP), dWh = tile_desc(smem_u32(sWh)), dWi = tile_desc(smem_u32(sWi));
    const uint64_t dD = N == 32 ? narrow_desc(usH + (TWICE ? 2 : 1) * buf) : tile_desc(usH + (TWICE ? 2 : 1) * buf);

    unsigned mb = 0u, phase = 0u;
#pragma unroll 1
    for (int step = s0; step < s_end; ++step) {
        // The tensor pipe holds the issuing warp until it has taken the products.  Two tiles per CTA: it hands its rows of sY over before,
        // so that the others' epilogues need not wait for its part of the next step's operands (n = m = 32, B = 16, T = 1e5: 1393 -> 1361
        // us per evaluation).  One tile: the products are what the step waits for, and go first (n = 64, m = 6: 1182 us, 1308 so).
        constexpr bool EARLY = N == 32 && TWICE;
        if constexpr (EARLY) {
            put_y();
            if (uwarp == 0) asm volatile("bar.arrive %0, %1;" ::"r"(1 + C::GROUPS + grp), "r"(C::GT) : "memory");
            else asm volatile("bar.arrive %0, %1;" ::"r"(1 + 2 * C::GROUPS + grp), "r"(C::GT) : "memory");
        }
        if (uwarp == 0) {
            tile_fence_after();
            if (tile_elect()) {
                const uint64_t at = TWICE && ((step - s0) & 1) ? (uint64_t)(buf >> 4) : 0ull, dH = dH0 + at, dX = dX0 + at;
                // x: hi hi, lo hi, hi lo into r z un
                for (int k = 0; k < kx; k += 16) {
                    tile_mma(utmem + N, dX + panel_k(128, k), dWi + panel_k(WR, k), tile_idesc(3 * N), k ? 1u : 0u);
                    tile_mma(utmem + N, dX + panel_k(128, kx + k), dWi + panel_k(WR, k), tile_idesc(3 * N), 1u);
                    tile_mma(utmem + N, dX + panel_k(128, k), dWi + panel_k(WR, kx + k), tile_idesc(3 * N), 1u);
                }
                // y: the same into q r z (q starts here)
                tile_mma(utmem, dH, dWh, tile_idesc(N), 0u);
                tile_mma(utmem + N, dH, dWh + ((N * 128) >> 4), tile_idesc(2 * N), 1u);
#pragma unroll
                for (int k = 0; k < N; k += 16) {
                    if (k) tile_mma(utmem, dH + panel_k(128, k), dWh + panel_k(WR, k), tile_idesc(3 * N), 1u);
                    tile_mma(utmem, dH + panel_k(128, N + k), dWh + panel_k(WR, k), tile_idesc(3 * N), 1u);
                    tile_mma(utmem, dH + panel_k(128, k), dWh + panel_k(WR, N + k), tile_idesc(3 * N), 1u);
                }
                // d
#pragma unroll
                for (int k = 0; k < N; k += 16)
                    tile_mma(utmem + 4 * N, dD + (uint64_t)(k >> 3), dWh + panel_k(WR, k), tile_idesc(3 * N), k ? 1u : 0u);
                tile_commit(&s_bar);
            }
            __syncwarp();
        }
        // the iterate of this step: for the owners' residual, and as the y operand of the next step; x of the next step
        if constexpr (!EARLY) put_y();
        const unsigned other = TWICE && ((step - s0) & 1) == 0 ? buf : 0u;
        if (TWICE) {
            put_h(sH + other);
            put_x(sX + other);
            load_y(step + 1);
            load_x(step + 2);
        }
        if (step == burn && own.te > 0) {                // what this chain assumed at its first own position
#pragma unroll
            for (int j = 0; j < 4; ++j)
                __stcg(reinterpret_cast<float4 *>(a.starts + gid * N + c0) + j, make_float4(d[2 * j].x, d[2 * j].y, d[2 * j + 1].x, d[2 * j + 1].y));
        }
        if constexpr (EARLY) {
            if (uwarp == 0) asm volatile("bar.sync %0, %1;" ::"r"(1 + 2 * C::GROUPS + grp), "r"(C::GT) : "memory");
            else asm volatile("bar.sync %0, %1;" ::"r"(1 + C::GROUPS + grp), "r"(C::GT) : "memory");
        } else {
            group_sync();
        }
        // (where it runs out, this step goes on with what it finds, and nothing of it counts)
        if (a.expire || !tile_wait(&s_bar, phase)) s_abort = 1;
        phase ^= 1u;
        tile_fence_after();
        if (!TWICE) {                                    // (the products are done with the operands)
            put_h(sH);
            put_x(sX);
            load_y(step + 1);
            load_x(step + 2);
        }

        const int t = own.ts + step;
        const bool act = t >= 0 && t < own.te, keep = act && step >= burn;
        float *yo = ynew + (ptrdiff_t)(own.e + step) * N + c0;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            float2 yn8[4];
            uint4 dp;
#pragma unroll
            for (int quad = 0; quad < 2; ++quad) {
                const int c = 8 * half + 4 * quad;       // columns c0 + c .. + 3
                float2 aq[2], ar[2], az_[2], an_[2], un[2], ur[2], uz[2];
                tile_ld4(tacc + c, aq);
                tile_ld4(tacc + N + c, ar);
                tile_ld4(tacc + 2 * N + c, az_);
                tile_ld4(tacc + 3 * N + c, an_);
                tile_ld4(tacc + 4 * N + c, un);
                tile_ld4(tacc + 5 * N + c, ur);
                tile_ld4(tacc + 6 * N + c, uz);
                const float4 bR4 = *reinterpret_cast<const float4 *>(sb + c0 + c), bZ4 = *reinterpret_cast<const float4 *>(sb + N + c0 + c);
                const float4 bQ4 = *reinterpret_cast<const float4 *>(sb + 2 * N + c0 + c), bN4 = *reinterpret_cast<const float4 *>(sb + 3 * N + c0 + c);
                const float4 y4 = *reinterpret_cast<const float4 *>(sY + row * C::YS + c0 + c);
                tile_wait_ld();
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const int j = (c >> 1) + p;
                    const float2 one = make_float2(1.0f, 1.0f), mone = make_float2(-1.0f, -1.0f);
                    const float2 bR = p ? make_float2(bR4.z, bR4.w) : make_float2(bR4.x, bR4.y), bZ = p ? make_float2(bZ4.z, bZ4.w) : make_float2(bZ4.x, bZ4.y);
                    const float2 bQ = p ? make_float2(bQ4.z, bQ4.w) : make_float2(bQ4.x, bQ4.y), bN = p ? make_float2(bN4.z, bN4.w) : make_float2(bN4.x, bN4.y);
                    const float2 y2 = p ? make_float2(y4.z, y4.w) : make_float2(y4.x, y4.y);
                    const float kE = -LOG2E * kS;
                    // r and z share a reciprocal; their exponentials are held below 2^60, so that the product stays finite
                    const float2 tr = ffma2(ar[p], make_float2(kE, kE), bR), tz = ffma2(az_[p], make_float2(kE, kE), bZ);
                    const float2 er = fadd2(make_float2(ex2_approx(min_nan(tr.x)), ex2_approx(min_nan(tr.y))), one);
                    const float2 ez = fadd2(make_float2(ex2_approx(min_nan(tz.x)), ex2_approx(min_nan(tz.y))), one);
                    const float2 ee = fmul2(er, ez), R = make_float2(rcp_approx(ee.x), rcp_approx(ee.y));
                    const float2 r = fmul2(R, ez), z = fmul2(R, er);
                    const float2 q = ffma2(aq[p], make_float2(kS, kS), bQ);
                    const float2 ac = ffma2(r, q, ffma2(an_[p], make_float2(kS, kS), bN));
                    const float2 t2 = fmul2(ac, make_float2(2.0f * LOG2E, 2.0f * LOG2E));
                    const float2 ec = fadd2(make_float2(ex2_approx(t2.x), ex2_approx(t2.y)), one);
                    const float2 cc = ffma2(make_float2(rcp_approx(ec.x), rcp_approx(ec.y)), make_float2(-2.0f, -2.0f), one);     // tanh
                    const float2 omz = ffma2(z, mone, one), omr = ffma2(r, mone, one);
                    const float2 hc = ffma2(cc, mone, hv[j]);
                    const float2 f = ffma2(z, hc, cc);
                    const float2 kz = fmul2(fmul2(z, omz), hc);
                    const float2 kn = fmul2(fmul2(omz, ffma2(fmul2(cc, mone), cc, one)), r);
                    const float2 kr = fmul2(fmul2(kn, q), omr);
                    const float2 s = ffma2(kr, ur[p], ffma2(kz, uz[p], fmul2(kn, un[p])));
                    const float2 yn = ffma2(s, make_float2(kD, kD), ffma2(z, d[j], f));
                    const float2 v = ffma2(y2, mone, yn);
                    if (keep) mb = max(mb, max(__float_as_uint(fabsf(v.x)), __float_as_uint(fabsf(v.y))));
                    d[j] = make_float2(act ? v.x : d[j].x, act ? v.y : d[j].y);
                    yn8[2 * quad + p] = yn;
                    hv[j] = y2;
                    const unsigned w = pack_f16(fmul2(d[j], make_float2(TILE_D_SCALE, TILE_D_SCALE)));
                    if (quad == 0) { if (p == 0) dp.x = w; else dp.y = w; } else { if (p == 0) dp.z = w; else dp.w = w; }
                }
            }
            if (keep) st_global_v8(yo + 8 * half, make_float4(yn8[0].x, yn8[0].y, yn8[1].x, yn8[1].y), make_float4(yn8[2].x, yn8[2].y, yn8[3].x, yn8[3].y));
            *reinterpret_cast<uint4 *>(sD + d_off(row, c0 + 8 * half)) = dp;
        }
        fence_proxy_async();
        tile_fence_before();
        group_sync();
        if (*(volatile int *)&s_abort) break;
    }

    // ---- boundaries: this row's end state against what its successor assumed
    unsigned mis = 0u;
    group_sync();
    if (has_next && row + 1 < C::ROWS) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 v = __ldcg(reinterpret_cast<const float4 *>(a.starts + (gid + 1) * N + c0) + j);
            mis = max(mis, max(max(absdiff_bits(v.x, d[2 * j].x), absdiff_bits(v.y, d[2 * j].y)), max(absdiff_bits(v.z, d[2 * j + 1].x), absdiff_bits(v.w, d[2 * j + 1].y))));
        }
    }
    if (row == C::ROWS - 1 && has_next) {                // the boundary behind this tile: side 0 of edge `tile`
        float *slot = a.edge + (size_t)tile * 2 * N + c0;
#pragma unroll
        for (int j = 0; j < 8; ++j) { __stcg(slot + 2 * j, d[j].x); __stcg(slot + 2 * j + 1, d[j].y); }
        s_side[0] = 1;
        __threadfence();
    }
    if (row == 0 && has_prev && tile > 0) {        // ... and the one before it: side 1 of edge tile - 1
        float *slot = a.edge + (size_t)(tile - 1) * 2 * N + N + c0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 v = __ldcg(reinterpret_cast<const float4 *>(a.starts + gid * N + c0) + j);
            __stcg(slot + 4 * j, v.x); __stcg(slot + 4 * j + 1, v.y); __stcg(slot + 4 * j + 2, v.z); __stcg(slot + 4 * j + 3, v.w);
        }
        s_side[1] = 1;
        __threadfence();
    }
    group_sync();
    if (warp < 2 && s_side[warp]) {
        const size_t edge = (size_t)tile - warp;
        unsigned old = 0;
        if (lane == 0) { __threadfence(); old = atomicAdd(a.edge_flag + edge, 1u); }
        old = __shfl_sync(0xffffffffu, old, 0);
        if (old == 1u) {
            __threadfence();
            const float *slot = a.edge + edge * 2 * N;
            for (int i = lane; i < N; i += 32) mis = max(mis, absdiff_bits(__ldcg(slot + i), __ldcg(slot + N + i)));
            if (lane == 0) a.edge_flag[edge] = 0u;
        }
    }
    mb = __reduce_max_sync(0xffffffffu, mb);
    mis = __reduce_max_sync(0xffffffffu, mis);
    if (lane == 0) {
        if (mb) atomicMax(&st->err_bits, mb);
        if (mis) atomicMax(&st->mis_bits, mis);
        __threadfence();
    }
    if (s_abort && tid == 0) {                           // a wait for the tensor core ran out: let what is in flight end
        tile_wait(&s_bar, phase ^ 1u);
        atomicOr(&st->flags, FLAG_TIMEOUT);
        __threadfence();
    }
    tile_fence_before();
    __syncthreads();
    tile_fence_after();
    if (all < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(C::TMEM) : "memory");
    if (all == 0) {
        __threadfence();
        const unsigned prev = atomicAdd(&st->exit_counter, 1u);
        if (prev + 1u == gridDim.x) {
            __threadfence();
            st->exit_counter = 0u;
            if (*(volatile unsigned *)&st->flags & FLAG_TIMEOUT) {         // rows that were not finished: nothing counts
                st->err_bits = 0u; st->mis_bits = 0u;
                st->done = BODY_TIMED_OUT;
                if (HostResult *h = st->host) post_done(h, BODY_TIMED_OUT);
            } else {
                body_decide(st, a, 1, BODY_ROUNDING, true);
            }
        }
    }
}

}  // namespace deer
