// The gradient's adjoint solve for n = 64 as one launch: the algorithm of newton_adjoint.cuh (see there: chains in
// descending time with a burn-in and verified boundaries, mu_t = J_{t+1}^T lambda_{t+1} as the state) with 128 chains in
// lockstep as the rows of a tcgen05 tile, in the manner of newton_tile.cuh.
//
// Per step and tile:
//   products 1   x_t W_i^T and y_{t-1} W_h^T, f16 hi + lo operands, three products each                  -> q r z un
//   epilogue 1   gates, lambda = gy + mu, the pre-activation gradients p = (p_r, p_z, p_n) (and p_a, the input side of the
//                third): to memory, and p as hi + lo f16 into tensor memory
//   products 2   p W_h, A from tensor memory, B = W_h's own operand read MN-major, three products           -> mu
// lambda has no natural scale (a mean over a long sequence, a loss on the last step only), so p carries a power of two per
// row and step, from the row's largest |lambda|.
// The pre-activation gradients leave as [position][4n] = (r, z, n hidden, n input): the two that dW_h and dW_i share once.
//
// What bounds it: latency, as in newton_tile.cuh.  m = 64, 80,000 positions: issue slots 36 % used, special functions 17 %, tensor
// 22 %, DRAM 4 %; per instruction issued 2.8 warps wait for a load (tensor memory, global), 2.6 at one of a step's three barriers.
#pragma once
#include "newton_adjoint.cuh"
#include "newton_tile.cuh"

namespace deer {

struct TileAdj {
    static constexpr int N = 64, THREADS = 8 * N, ROWS = 128;
    static constexpr int CG = N / 16;                    // threads of a row
    static constexpr int LPR = N / 4, GS = N + 4;
    static constexpr unsigned PANEL = 128 * 128, HP = 2 * N / 64, WROWS = 3 * N;
    static constexpr unsigned TMEM = 512;                // columns: q r z un (n each), mu (n), p hi and lo (3n / 2 each)
    __host__ __device__ static constexpr unsigned xp(int kx) { return (2 * kx + 63) / 64; }
    static constexpr size_t smem(int kx)
    {
        return 1024 + (size_t)PANEL * (HP + xp(kx)) + (size_t)WROWS * 128 * (HP + xp(kx)) +
               sizeof(float) * (ROWS * GS + CG * ROWS + 4 * N) + sizeof(TileRow) * ROWS;
    }
};

__global__ void __launch_bounds__(TileAdj::THREADS, 1) adjoint_tile_kernel(AdjArgs a)
{
    using C = TileAdj;
    constexpr int N = C::N;
    constexpr unsigned WR = C::WROWS;
    constexpr float LOG2E = 1.4426950408889634f;
    StatusBlock *st = a.st;
    const int burn = adjoint_burn(a, st);
    if (*(volatile int *)&st->done || burn == 0) return;

    extern __shared__ __align__(16) unsigned char smem_tile[];
    __shared__ __align__(8) uint64_t bar1, bar2;
    __shared__ unsigned s_tmem, s_top;
    __shared__ __align__(16) float s_xf[64];
    __shared__ int s_abort[2], s_side[2];               // s_abort: a wait for products 1, 2 ran out (each read behind a sync that
                                                         // follows its writes, and before one that precedes the next)
    unsigned char *sm = (unsigned char *)(((uintptr_t)smem_tile + 1023) & ~(uintptr_t)1023);
    const int m = a.m, kx = (m + 15) & ~15;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned char *sWh = sm, *sWi = sWh + WR * 128 * C::HP;
    unsigned char *sH = sWi + WR * 128 * C::xp(kx), *sX = sH + C::PANEL * C::HP;
    float *sb = reinterpret_cast<float *>(sX + C::PANEL * C::xp(kx));
    float *sG = sb + 4 * N, *sMax = sG + C::ROWS * C::GS;
    TileRow *rows = reinterpret_cast<TileRow *>(sMax + C::CG * C::ROWS);
    const int L = a.L, T = a.T, nchain = (T + L - 1) / L;
    const long long total = (long long)a.B * nchain;
    const long long tile = blockIdx.x;

    // ---- weights, biases, geometry, tensor memory
    const float wscale = operand_scales(a.h0.W_h, a.h0.W_i, 3 * N, N, m, TILE_OP_SCALE, TILE_TOP, s_xf, &s_top);
    const float unit = wscale * TILE_OP_SCALE, kS = 1.0f / unit;
    for (int i = tid; i < (int)WR * (N / 2); i += C::THREADS) {          // rows of W_h in the order n, r, z
        const int k = 2 * (i % (N / 2)), r = i / (N / 2), gate = r < N ? 2 : r / N - 1;
        const float2 v = *reinterpret_cast<const float2 *>(a.h0.W_h + (size_t)(gate * N + r % N) * N + k);
        unsigned hi, lo;
        split_f16(make_float2(v.x * wscale, v.y * wscale), hi, lo);
        *reinterpret_cast<unsigned *>(sWh + panel_off(WR, r, k)) = hi;
        *reinterpret_cast<unsigned *>(sWh + panel_off(WR, r, N + k)) = lo;
    }
    for (int i = tid; i < (int)WR * (kx / 2); i += C::THREADS) {         // rows of W_i in the order r, z, n
        const int k = 2 * (i % (kx / 2)), r = i / (kx / 2);
        const float *w = a.h0.W_i + (size_t)r * m + k;
        unsigned hi, lo;
        split_f16(make_float2(k < m ? w[0] * (unit * pow2_inverse(s_xf[k])) : 0.0f, k + 1 < m ? w[1] * (unit * pow2_inverse(s_xf[k + 1])) : 0.0f), hi, lo);
        *reinterpret_cast<unsigned *>(sWi + panel_off(WR, r, k)) = hi;
        *reinterpret_cast<unsigned *>(sWi + panel_off(WR, r, kx + k)) = lo;
    }
    for (int i = tid; i < N; i += C::THREADS) {
        sb[i] = -LOG2E * (a.h0.b_h[i] + a.h0.b_i[i]);
        sb[N + i] = -LOG2E * (a.h0.b_h[N + i] + a.h0.b_i[N + i]);
        sb[2 * N + i] = a.h0.b_h[2 * N + i];
        sb[3 * N + i] = a.h0.b_i[2 * N + i];
    }
    if (tid < C::ROWS) {                                 // scan position q of a sequence is time step T - 1 - q
        const long long gid = tile * C::ROWS + tid;
        TileRow r{0, 0, 0, 0};
        if (gid < total) {
            const long long b = gid / nchain;
            const int c = (int)(gid - b * nchain);
            r.ts = c * L - burn;
            r.te = min(T, (c + 1) * L);
            r.e = (int)(b * T + T - 1 - r.ts);
            r.b = (int)b;
        }
        rows[tid] = r;
    }
    if (tid == 0) { mbar_init(&bar1, 1); mbar_init(&bar2, 1); s_abort[0] = s_abort[1] = 0; s_side[0] = s_side[1] = 0; }
    if (tid < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(C::TMEM) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tile_fence_before();
    __syncthreads();
    tile_fence_after();
    const unsigned tmem = s_tmem;
    const int xv = (m & 3) == 0 && ((uintptr_t)a.x & 15) == 0 ? 4 : (m & 1) == 0 && ((uintptr_t)a.x & 7) == 0 ? 2 : 1;

    // ---- loader mapping: rows lr + 32 i, columns 4 lc .. 4 lc + 3
    const int lr = tid / C::LPR, lc = tid % C::LPR;
    float4 yv[4], xr[4];
    unsigned x_in = 0u;                                  // rows (bit i) that are inside their chain
    auto load = [&](int step) {                          // the state before every row's time step, and x there
        x_in = 0u;
        const float *p[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const TileRow r = rows[lr + 32 * i];
            const int q = r.ts + step;
            const bool in = q >= 0 && q < r.te, first = q == T - 1;
            x_in |= (in ? 1u : 0u) << i;
            p[i] = a.x + (size_t)(unsigned)(in ? r.e - step : 0) * m;
            const float *h = (in && !first ? a.y : a.y0) + (size_t)(unsigned)(in && !first ? r.e - step - 1 : r.b) * N;
            yv[i] = __ldg(reinterpret_cast<const float4 *>(h) + lc);
        }
        const int c = 4 * lc;
        if (xv == 4) {
            const int cc = min(c, m - 4);
#pragma unroll
            for (int i = 0; i < 4; ++i) xr[i] = __ldg(reinterpret_cast<const float4 *>(p[i] + cc));
        } else if (xv == 2) {
            const int ca = min(c, m - 2), cb = min(c + 2, m - 2);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 u = __ldg(reinterpret_cast<const float2 *>(p[i] + ca)), v = __ldg(reinterpret_cast<const float2 *>(p[i] + cb));
                xr[i] = make_float4(u.x, u.y, v.x, v.y);
            }
        } else {
            const int c1 = min(c, m - 1), c2 = min(c + 1, m - 1), c3 = min(c + 2, m - 1), c4 = min(c + 3, m - 1);
#pragma unroll
            for (int i = 0; i < 4; ++i) xr[i] = make_float4(__ldg(p[i] + c1), __ldg(p[i] + c2), __ldg(p[i] + c3), __ldg(p[i] + c4));
        }
    };
    // dL/dy of every row's step straight into sG (zeros outside the chain); where it is the same at all steps, once, whole
    auto load_g = [&](int step) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const TileRow r = rows[lr + 32 * i];
            const int q = r.ts + step;
            const bool in = q >= 0 && q < r.te;
            const float *src = (a.gy_seq ? a.gy_seq + (size_t)(unsigned)r.b * N : a.gy + (size_t)(unsigned)(in ? r.e - step : 0) * N) + 4 * lc;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(sG + (lr + 32 * i) * C::GS + 4 * lc)), "l"(src), "r"(in || a.gy_seq ? 16 : 0) : "memory");
        }
        cp_async_commit();
    };
    auto put = [&](unsigned char *panel, int row, int k, int klo, float4 v, float4 f) {
        uint2 hi, lo;
        split_f16(fmul2(make_float2(v.x, v.y), make_float2(f.x, f.y)), hi.x, lo.x);
        split_f16(fmul2(make_float2(v.z, v.w), make_float2(f.z, f.w)), hi.y, lo.y);
        *reinterpret_cast<uint2 *>(panel + panel_off(128, row, k)) = hi;
        *reinterpret_cast<uint2 *>(panel + panel_off(128, row, klo + k)) = lo;
    };
    auto wanted = [](bool in, float4 v) { return in ? v : make_float4(0.f, 0.f, 0.f, 0.f); };
    const bool whole = (m & 3) == 0;
    auto put_operands = [&]() {
#pragma unroll
        for (int i = 0; i < 4; ++i) put(sH, lr + 32 * i, 4 * lc, N, wanted((x_in >> i) & 1u, yv[i]), make_float4(TILE_OP_SCALE, TILE_OP_SCALE, TILE_OP_SCALE, TILE_OP_SCALE));
        const int c = 4 * lc;
        if (c >= kx) return;
        const float4 f = *reinterpret_cast<const float4 *>(s_xf + c);       // (the channels' units, whatever they are: 888 -> 895 us at m = 64, 320,000 positions)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float4 v = wanted((x_in >> i) & 1u && c < m, xr[i]);
            if (!whole) { v.y = c + 1 < m ? v.y : 0.f; v.z = c + 2 < m ? v.z : 0.f; v.w = c + 3 < m ? v.w : 0.f; }
            put(sX, lr + 32 * i, c, kx, v, f);
        }
    };

    // ---- owner mapping: row and 16 columns of this thread
    const int row = (warp & 3) * 32 + lane, cg = warp >> 2, c0 = cg * 16;
    const TileRow own = rows[row];
    const long long gid = tile * C::ROWS + row;
    const unsigned tacc = tmem + ((unsigned)(32 * (warp & 3)) << 16);
    const int chain = (int)(gid % nchain);
    const bool has_next = own.te > 0 && chain + 1 < nchain, has_prev = own.te > 0 && chain > 0;
    float2 d[8];                                         // mu
#pragma unroll
    for (int j = 0; j < 8; ++j) d[j] = make_float2(0.f, 0.f);
    const int s0 = nchain == 1 ? burn : 0, s_end = tile * C::ROWS < total ? burn + min(L, T) : s0;      // (a tile without rows: no steps)

    load(s0);
    load_g(s0);
    put_operands();

    // warp-uniform copies for the issuing warp
    const int uwarp = __shfl_sync(0xffffffffu, warp, 0);
    const unsigned utmem = __shfl_sync(0xffffffffu, tmem, 0), usH = __shfl_sync(0xffffffffu, smem_u32(sH), 0);
    const uint64_t dH = tile_desc(usH), dX = tile_desc(usH + C::PANEL * C::HP), dWh = tile_desc(smem_u32(sWh)), dWi = tile_desc(smem_u32(sWi));

    unsigned mb = 0u, phase = 0u, mb_end = 0u;          // mb: the row's largest |lambda|, from the window on
    float scale = 0.0f;                                  // ... over the window: of the boundary before this chain
#pragma unroll 1
    for (int step = s0; step < s_end; ++step) {
        if (step == burn - ADJ_WINDOW) mb = 0u;
        if (step == burn) scale = __uint_as_float(mb);
        if (step == burn && own.te > 0) {                // what this chain assumed at its first own position
#pragma unroll
            for (int j = 0; j < 4; ++j)
                __stcg(reinterpret_cast<float4 *>(a.starts + gid * N + c0) + j, make_float4(d[2 * j].x, d[2 * j].y, d[2 * j + 1].x, d[2 * j + 1].y));
        }
        const int q = own.ts + step;
        const bool act = q >= 0 && q < own.te, keep = act && step >= burn;
        cp_async_wait_0();
        fence_proxy_async();
        tile_fence_before();
        __syncthreads();                                    // operands and dL/dy of this step are there
        if (*(volatile int *)&s_abort[1]) break;
        // ---- lambda = gy + mu, and the row's scale (the other threads of the row have the other columns)
        float2 l[8];
        unsigned top = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float4 g4 = *reinterpret_cast<const float4 *>(sG + row * C::GS + c0 + 4 * j);
            if (a.gy_seq && !act) g4 = make_float4(0.f, 0.f, 0.f, 0.f);
            l[2 * j] = fadd2(make_float2(g4.x, g4.y), d[2 * j]);
            l[2 * j + 1] = fadd2(make_float2(g4.z, g4.w), d[2 * j + 1]);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) top = max(top, max(__float_as_uint(fabsf(l[j].x)), __float_as_uint(fabsf(l[j].y))));
        sMax[cg * C::ROWS + row] = __uint_as_float(top);
        // Products 1, and the rows' maxima for everybody.  The pipe holds the issuing warp until its last product (2,400 cycles at
        // m = 64), so it does not hold the others: it arrives before it issues, and waits for the others' maxima behind
        // (m = 64, 575,000 positions: 852 -> 775 us; with one barrier the next step's loads began behind the products).
        if (uwarp == 0) {
            asm volatile("bar.arrive 1, %0;" ::"r"(C::THREADS) : "memory");
            tile_fence_after();
            if (tile_elect()) {
                for (int k = 0; k < kx; k += 16) {       // x: hi hi, lo hi, hi lo into r z un
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
                tile_commit(&bar1);
            }
            __syncwarp();
            asm volatile("bar.sync 2, %0;" ::"r"(C::THREADS) : "memory");
        } else {
            asm volatile("bar.arrive 2, %0;" ::"r"(C::THREADS) : "memory");
            asm volatile("bar.sync 1, %0;" ::"r"(C::THREADS) : "memory");
        }
#pragma unroll
        for (int k = 0; k < C::CG; ++k) top = max(top, __float_as_uint(sMax[k * C::ROWS + row]));
        mb = max(mb, top);                                  // (outside the chain: zero, or what it ended with)
        // p up to about 2^8 (|p| <= |lambda| / 4 or so): exponent of the row's largest |lambda| to 2^9
        const int ex = min(max((int)(top >> 23), 20), 240);
        const float sc = __uint_as_float((unsigned)(127 + 9 - (ex - 127)) << 23), inv = __uint_as_float((unsigned)(127 - 9 + (ex - 127)) << 23);
        const float kM = inv / wscale;
        if (step + 1 < s_end) {
            load(step + 1);
            if (!a.gy_seq) load_g(step + 1);
        }
        if (a.expire || !tile_wait(&bar1, phase)) s_abort[0] = 1;
        tile_fence_after();
        // ---- gates, pre-activation gradients
        float *go = a.dGi + (ptrdiff_t)(own.e - step) * (4 * N) + c0;
        const float2 one = make_float2(1.0f, 1.0f), mone = make_float2(-1.0f, -1.0f);
        const float kE = -LOG2E * kS;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            float2 pr8[4], pz8[4], pn8[4], pa8[4];
            const uint4 hh = *reinterpret_cast<const uint4 *>(sH + panel_off(128, row, c0 + 8 * half)), hl = *reinterpret_cast<const uint4 *>(sH + panel_off(128, row, N + c0 + 8 * half));
#pragma unroll
            for (int quad = 0; quad < 2; ++quad) {
                const int c = c0 + 8 * half + 4 * quad;  // columns c .. c + 3
                float2 aq[2], ar[2], az_[2], an_[2];
                tile_ld4(tacc + c, aq);
                tile_ld4(tacc + N + c, ar);
                tile_ld4(tacc + 2 * N + c, az_);
                tile_ld4(tacc + 3 * N + c, an_);
                const float4 bR4 = *reinterpret_cast<const float4 *>(sb + c), bZ4 = *reinterpret_cast<const float4 *>(sb + N + c);
                const float4 bQ4 = *reinterpret_cast<const float4 *>(sb + 2 * N + c), bN4 = *reinterpret_cast<const float4 *>(sb + 3 * N + c);
                tile_wait_ld();
                unsigned hi[3][2], lo[3][2];
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const int j = 4 * half + 2 * quad + p;
                    const float2 bR = p ? make_float2(bR4.z, bR4.w) : make_float2(bR4.x, bR4.y), bZ = p ? make_float2(bZ4.z, bZ4.w) : make_float2(bZ4.x, bZ4.y);
                    const float2 bQ = p ? make_float2(bQ4.z, bQ4.w) : make_float2(bQ4.x, bQ4.y), bN = p ? make_float2(bN4.z, bN4.w) : make_float2(bN4.x, bN4.y);
                    const unsigned wh = quad == 0 ? (p ? hh.y : hh.x) : (p ? hh.w : hh.z), wl = quad == 0 ? (p ? hl.y : hl.x) : (p ? hl.w : hl.z);
                    const float2 h2 = fmul2(fadd2(__half22float2(*reinterpret_cast<const __half2 *>(&wh)), __half22float2(*reinterpret_cast<const __half2 *>(&wl))),
                                            make_float2(1.0f / TILE_OP_SCALE, 1.0f / TILE_OP_SCALE));
                    const float2 tr = ffma2(ar[p], make_float2(kE, kE), bR), tz = ffma2(az_[p], make_float2(kE, kE), bZ);
                    const float2 er = fadd2(make_float2(ex2_approx(min_nan(tr.x)), ex2_approx(min_nan(tr.y))), one);
                    const float2 ez = fadd2(make_float2(ex2_approx(min_nan(tz.x)), ex2_approx(min_nan(tz.y))), one);
                    const float2 ee = fmul2(er, ez), R = make_float2(rcp_approx(ee.x), rcp_approx(ee.y));
                    const float2 r = fmul2(R, ez), z = fmul2(R, er);
                    const float2 qn = ffma2(aq[p], make_float2(kS, kS), bQ);
                    const float2 ac = ffma2(r, qn, ffma2(an_[p], make_float2(kS, kS), bN));
                    const float2 t2 = fmul2(ac, make_float2(2.0f * LOG2E, 2.0f * LOG2E));
                    const float2 ec = fadd2(make_float2(ex2_approx(t2.x), ex2_approx(t2.y)), one);
                    const float2 cc = ffma2(make_float2(rcp_approx(ec.x), rcp_approx(ec.y)), make_float2(-2.0f, -2.0f), one);     // tanh
                    const float2 omz = ffma2(z, mone, one), omr = ffma2(r, mone, one);
                    const float2 lz = fmul2(z, l[j]), lo2 = fmul2(omz, l[j]);
                    const float2 pz = fmul2(fmul2(lo2, z), ffma2(cc, mone, h2));
                    const float2 pa = fmul2(lo2, ffma2(fmul2(cc, mone), cc, one));
                    const float2 pn = fmul2(pa, r);
                    const float2 pr = fmul2(fmul2(pn, qn), omr);
                    l[j] = lz;
                    pr8[2 * quad + p] = pr; pz8[2 * quad + p] = pz; pn8[2 * quad + p] = pn; pa8[2 * quad + p] = pa;
                    const float2 s2 = make_float2(sc, sc);
                    split_f16(fmul2(pn, s2), hi[0][p], lo[0][p]);                   // (the order of W_h's rows: n, r, z)
                    split_f16(fmul2(pr, s2), hi[1][p], lo[1][p]);
                    split_f16(fmul2(pz, s2), hi[2][p], lo[2][p]);
                }
#pragma unroll
                for (int g = 0; g < 3; ++g) {
                    tile_st2(tacc + 5 * N + (g * N + c) / 2, hi[g][0], hi[g][1]);
                    tile_st2(tacc + 5 * N + (3 * N + g * N + c) / 2, lo[g][0], lo[g][1]);
                }
            }
            if (keep) {
                auto st8 = [&](float *o, const float2 (&v)[4]) { st_global_v8(o, make_float4(v[0].x, v[0].y, v[1].x, v[1].y), make_float4(v[2].x, v[2].y, v[3].x, v[3].y)); };
                st8(go + 8 * half, pr8); st8(go + N + 8 * half, pz8); st8(go + 2 * N + 8 * half, pn8); st8(go + 3 * N + 8 * half, pa8);
            }
        }
        tile_wait_st();
        tile_fence_before();
        __syncthreads();                                    // p of every row is in tensor memory; the operands are free
        if (*(volatile int *)&s_abort[0]) break;
        if (uwarp == 0) {
            tile_fence_after();
            if (tile_elect()) {
                // p W_h: K steps of 16 gate rows; B MN-major: 16 rows of W_h's operand, n contiguous (lo half: n f16 further on)
                const uint64_t lo_at = (uint64_t)((WR * 128) >> 4);
#pragma unroll
                for (int k = 0; k < 3 * N; k += 16) {
                    const uint64_t b = dWh + (uint64_t)((k * 128) >> 4);
                    tile_mma_ta(utmem + 4 * N, utmem + 5 * N + k / 2, b, tile_idesc(N) | TILE_B_MN, k ? 1u : 0u);
                    tile_mma_ta(utmem + 4 * N, utmem + 5 * N + 3 * N / 2 + k / 2, b, tile_idesc(N) | TILE_B_MN, 1u);
                    tile_mma_ta(utmem + 4 * N, utmem + 5 * N + k / 2, b + lo_at, tile_idesc(N) | TILE_B_MN, 1u);
                }
                tile_commit(&bar2);
            }
            __syncwarp();
        }
        if (step + 1 < s_end) put_operands();
        if (!tile_wait(&bar2, phase)) s_abort[1] = 1;
        phase ^= 1u;
        tile_fence_after();
#pragma unroll
        for (int quad = 0; quad < 4; ++quad) {
            float2 am[2];
            tile_ld4(tacc + 4 * N + c0 + 4 * quad, am);
            tile_wait_ld();
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const float2 v = ffma2(am[p], make_float2(kM, kM), l[2 * quad + p]);
                d[2 * quad + p] = make_float2(act ? v.x : d[2 * quad + p].x, act ? v.y : d[2 * quad + p].y);
            }
        }
    }
    cp_async_wait_0();
    __syncthreads();
    if (cg == 0) sMax[row] = scale;
    __syncthreads();

    // ---- the state that leaves the first time step: the gradient w.r.t. y0.  Wanted or not, it shows an input beyond f16's range
    // at that step, which reaches no boundary.
    if (own.te > 0 && !has_next) {
#pragma unroll
        for (int j = 0; j < 8; ++j) mb_end = max(mb_end, max(__float_as_uint(fabsf(d[j].x)), __float_as_uint(fabsf(d[j].y))));
        if (a.dy0) {
            float *o = a.dy0 + (size_t)own.b * N + c0;
#pragma unroll
            for (int j = 0; j < 8; ++j) { o[2 * j] = d[j].x; o[2 * j + 1] = d[j].y; }
        }
    }
    // ---- boundaries: this row's end state against what its successor assumed
    const int reach = DY0_REACH * burn;
    unsigned mis = 0u, rel = 0u, mis_end = 0u;
    if (has_next && row + 1 < C::ROWS) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 v = __ldcg(reinterpret_cast<const float4 *>(a.starts + (gid + 1) * N + c0) + j);
            mis = max(mis, max(max(absdiff_bits(v.x, d[2 * j].x), absdiff_bits(v.y, d[2 * j].y)), max(absdiff_bits(v.z, d[2 * j + 1].x), absdiff_bits(v.w, d[2 * j + 1].y))));
        }
        rel = boundary_ratio(mis, sMax[row + 1]);
        if (T - own.te < reach) mis_end = mis;
    }
    if (row == C::ROWS - 1 && has_next) {                // the boundary behind this tile: side 0 of edge `tile`
        float *slot = a.edge + (size_t)tile * ADJ_EDGE(N) + c0;
#pragma unroll
        for (int j = 0; j < 8; ++j) { __stcg(slot + 2 * j, d[j].x); __stcg(slot + 2 * j + 1, d[j].y); }
        s_side[0] = T - own.te < reach ? 2 : 1;
        __threadfence();
    }
    if (row == 0 && has_prev && tile > 0) {              // ... and the one before it: side 1 of edge tile - 1
        float *slot = a.edge + (size_t)(tile - 1) * ADJ_EDGE(N) + N + c0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 v = __ldcg(reinterpret_cast<const float4 *>(a.starts + gid * N + c0) + j);
            __stcg(slot + 4 * j, v.x); __stcg(slot + 4 * j + 1, v.y); __stcg(slot + 4 * j + 2, v.z); __stcg(slot + 4 * j + 3, v.w);
        }
        if (cg == 0) __stcg(slot + N, scale);
        s_side[1] = T - chain * L < reach ? 2 : 1;
        __threadfence();
    }
    __syncthreads();
    if (warp < 2 && s_side[warp]) {
        const size_t edge = (size_t)tile - warp;
        unsigned old = 0;
        if (lane == 0) { __threadfence(); old = atomicAdd(a.edge_flag + edge, 1u); }
        old = __shfl_sync(0xffffffffu, old, 0);
        if (old == 1u) {
            __threadfence();
            const float *slot = a.edge + edge * ADJ_EDGE(N);
            for (int i = lane; i < N; i += 32) {
                const unsigned q = absdiff_bits(__ldcg(slot + i), __ldcg(slot + N + i));
                mis = max(mis, q);
                rel = max(rel, boundary_ratio(q, __ldcg(slot + 2 * N)));
                if (s_side[warp] == 2) mis_end = max(mis_end, q);
            }
            if (lane == 0) a.edge_flag[edge] = 0u;
        }
    }
    mb = __reduce_max_sync(0xffffffffu, mb);
    mis = __reduce_max_sync(0xffffffffu, mis);
    rel = __reduce_max_sync(0xffffffffu, rel);
    mb_end = __reduce_max_sync(0xffffffffu, mb_end);
    mis_end = __reduce_max_sync(0xffffffffu, mis_end);
    if (lane == 0) {
        if (mb) atomicMax(&st->err_bits, mb);
        if (mis) atomicMax(&st->mis_bits, mis);
        if (rel) atomicMax(&st->rel_bits, rel);
        if (mb_end) atomicMax(&st->top_end_bits, mb_end);
        if (mis_end) atomicMax(&st->mis_end_bits, mis_end);
        __threadfence();
    }
    if ((s_abort[0] || s_abort[1]) && tid == 0) {                           // a wait for the tensor core ran out: let what is in flight end
        if (s_abort[0]) tile_wait(&bar1, phase); else tile_wait(&bar2, phase ^ 1u);
        atomicOr(&st->flags, FLAG_TIMEOUT);
        __threadfence();
    }
    tile_fence_before();
    __syncthreads();
    tile_fence_after();
    if (tid < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(C::TMEM) : "memory");
    if (tid == 0) {
        __threadfence();
        const unsigned prev = atomicAdd(&st->exit_counter, 1u);
        if (prev + 1u == gridDim.x) {
            __threadfence();
            st->exit_counter = 0u;
            adjoint_decide(st, a.eta, a.dy0 != nullptr, burn);
        }
    }
}

}  // namespace deer
