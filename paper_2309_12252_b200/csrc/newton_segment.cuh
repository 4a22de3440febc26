// One Newton body as one launch, for problems that do not fill the GPU with long chains and for all small states: the same
// solve as newton_body.cuh (chains with a burn-in, boundaries verified, see there), organised in two phases per CTA.
//
// In the one-phase kernel every step of a chain is a whole cell -- some thousand cycles in series, times burn + L steps --
// which is what a small problem takes whatever its size, and the burn-in's cells are evaluated twice.  Here a CTA owns NC
// consecutive chains, L positions each, of which a chain's burn-in are its predecessors' positions:
//   phase 1  the cell at every position of the CTA once, 16 positions per warp and MMA tile, nothing in series: residual and
//            coefficients {z, k_r, a_z, k_n, r} [5N] of a position stay in shared memory;
//   phase 2  the chains, 16 in lockstep per group of N / 8 warps (one block of eight state columns each), a step being
//            d <- r + z.d + k_r.(W_hr d) + a_z.(W_hz d) + k_n.(W_hn d):  9 MMAs of a warp per K step (of 16 columns of d, of
//            eight in TF32; 3 where products with d are single), the new d crossing to the other warps of the group
//            through shared memory, as the f16 halves of the next step's operand where products are on those.
// What bounds it: phases in series.  Cycles of a body, read with clock64 by one warp where burn-ins were 45 steps (n = 8, m = 4, B = 16,
// T = 1e4: 64 chains of 17 positions per CTA) and 30 (n = 4, m = 2, T = 1000: 16 chains of 5); they now follow the body, 24 ... 40 and 16
// ... 30.  n = 8: phase 1 10,250 (five tiles a warp), burn-in 170 a step, the 17 positions owned 10,800 (640 a step, with its old
// iterate, residual and store), prologue of phase 2 950, exchange with the other CTAs 4,000 ... 10,000.  n = 4: 3,500, 170 a step, 3,550,
// 1,200, 3,000.  Issue slots 34 % used; the warps that phase 2 has no chains for wait at the barrier behind it, 5.8 of 16 at a time.
#pragma once
#include "newton_body.cuh"

namespace deer {

template <int N, bool EXACT> struct Seg {
    static constexpr int NT = N / 8;
    // f16 halves, as in newton_body.cuh; TF32 for n <= 8, where a block of columns is half of a K step of 16, and for n = 16, whose
    // single products with the update gain less than the halves' conversions cost.  (us per evaluation, TF32 / f16: n = 24,
    // 20,000 positions 174 / 164, 8,000 100 / 96; n = 12, 96,000 289 / 281; n = 9, 2,700 78 / 76; n = 32, 16,000 106 / 104; n = 16,
    // 80,000 231 / 235, 16,000 88 / 90.)
    static constexpr bool F16 = NT > (EXACT ? 1 : 2);
    static constexpr int KB = F16 ? 2 : 1, NB = (NT + KB - 1) / KB;      // column blocks of a K step, K steps
    static constexpr int WARPS = N == 8 ? 16 : 8, THREADS = 32 * WARPS;
    static constexpr int GROUPS = NT >= 4 ? 1 : 4 / NT;  // groups of 16 chains at most: one warp of phase 2 per sub-partition (a second
                                                         // one there makes a step of exact products 1.9 times as long)
    static constexpr int NC_MAX = 16 * GROUPS;           // chains of a CTA
    static constexpr int NS = 3 * N + 2;
    static constexpr int SZ = 5 * N + (N % 16 == 0 ? 8 : 0);             // floats of a slot: = 8 or 24 (mod 32), so that with odd L
                                                         // eight rows L slots apart fall into distinct bank groups
    static constexpr int DS = N + (N % 16 == 0 ? 8 : 0);        // stride of an exchanged update
    static constexpr size_t fixed(int kx)                // weights, biases, chain table, start states, exchange buffers
    {
        return sizeof(float) * ((size_t)16 * (NB + (kx + KB - 1) / KB) * NS + 4 * N + (size_t)(NC_MAX + 1) * DS + (size_t)2 * NC_MAX * DS) + 32 * (size_t)NC_MAX;
    }
};

constexpr unsigned BODY_SPIN_LIMIT = 1u << 22;           // polls of a wait for another CTA (a second or two)

// {tag, bits} words: a value and the round it belongs to in one 64-bit store
__device__ __forceinline__ void st_relaxed_u64w(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void st_word(unsigned long long *p, int i, int n, float v, unsigned tag)
{
    if (i < n) st_relaxed_u64w(p + i, ((unsigned long long)tag << 32) | __float_as_uint(v));
}
__device__ __forceinline__ unsigned wait_word(const unsigned long long *p, unsigned tag, bool &gave_up)
{
    unsigned long long v = 0;
    for (unsigned spins = 0;; ++spins) {
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
        if ((unsigned)(v >> 32) == tag) break;
        if (spins > BODY_SPIN_LIMIT) { gave_up = true; break; }
    }
    return (unsigned)v;
}

struct SegChain { long long e; int t0, t_end, b, next; };      // e: row of position 0 in [B,T]; t0: first owned position
static_assert(sizeof(SegChain) <= 32, "chain table entry");

template <int N, bool V2, bool EXACT>
__global__ void __launch_bounds__(Seg<N, EXACT>::THREADS, 1) newton_segment_kernel(BodyArgs a, int NC, int whole_loop)
{
    using C = Seg<N, EXACT>;
    constexpr int NT = C::NT, KB = C::KB, NB = C::NB, NS = C::NS, SZ = C::SZ, DS = C::DS;
    constexpr bool F16 = C::F16;
    __shared__ unsigned s_top;
    __shared__ __align__(16) float s_xf[64];
    extern __shared__ __align__(16) float smb[];
    const BodyHead hd = a.heads ? a.heads[blockIdx.y] : a.h0;
    StatusBlock *st = a.st + blockIdx.y;
    const int n = a.n, m = a.m, H = a.H, L = a.L;
    const bool proj = a.u == nullptr;
    const int kx = proj ? (m + 8 * KB - 1) / (8 * KB) : 0;               // K steps of x
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t = lane & 3;

    const int s = hd.stride, Tp = (a.T + s - 1) / s, nchain = (Tp + L - 1) / L;
    const long long total = (long long)a.B * s * nchain;
    const unsigned nctas = (unsigned)((total + NC - 1) / NC);
    if (blockIdx.x >= nctas) return;

    uint4 *sH = reinterpret_cast<uint4 *>(smb), *sI = sH + 4 * NB * NS;
    float *sb = reinterpret_cast<float *>(sI + 4 * kx * NS);
    float *ss = sb + 4 * N;                              // start state of every chain, and of the one behind the last
    float *dx = ss + (C::NC_MAX + 1) * DS;               // exchanged updates [2][NC_MAX][DS]
    SegChain *tab = reinterpret_cast<SegChain *>(dx + 2 * C::NC_MAX * DS);
    float *slots = reinterpret_cast<float *>(tab + C::NC_MAX);
    float wscale = 1.0f, unit = 1.0f, kS = 1.0f, kD = 1.0f;
    if constexpr (F16) {
        wscale = operand_scales(hd.W_h, hd.W_i, 3 * n, n, proj ? m : 0, MMA_OP_SCALE, MMA_TOP, s_xf, &s_top);
        unit = wscale * MMA_OP_SCALE;
        kS = 1.0f / unit;
        kD = 1.0f / (wscale * MMA_D_SCALE);
    }
    // weights as records of the four words that a lane needs for a column of a K step (newton_body.cuh)
    auto record = [&](const float *wr, bool row, int kt, int width, auto scale) {
        const int k = 8 * KB * (kt >> 2) + 2 * (kt & 3);
        auto w = [&](int j) { return row && j < width ? wr[j] * scale(j) : 0.0f; };
        uint4 r;
        if constexpr (F16) {
            split_f16(make_float2(w(k), w(k + 1)), r.x, r.z);
            split_f16(make_float2(w(k + 8), w(k + 9)), r.y, r.w);
        } else {
            split_tf32(w(k), r.x, r.z);
            split_tf32(w(k + 1), r.y, r.w);
        }
        return r;
    };
    for (int idx = tid; idx < 4 * NB * 3 * N; idx += C::THREADS) {
        const int kt = idx % (4 * NB), c = idx / (4 * NB), gate = c / N, i = c % N;
        sH[kt * NS + c] = record(hd.W_h + (size_t)(gate * n + i) * n, i < n, kt, n, [&](int) { return wscale; });
    }
    for (int idx = tid; idx < 4 * kx * 3 * N; idx += C::THREADS) {
        const int kt = idx % (4 * kx), c = idx / (4 * kx), gate = c / N, i = c % N;
        sI[kt * NS + c] = record(hd.W_i + (size_t)(gate * n + i) * m, i < n, kt, m, [&](int j) { return F16 ? unit * pow2_inverse(s_xf[j]) : 1.0f; });
    }
    // block b of a K step of an A operand, row h of this lane: two columns (an accumulator's columns of TF32 in the slots t, t + 4)
    auto operand = [&](unsigned (&hi)[4], unsigned (&lo)[4], int b, int h, float2 v, float2 scale = make_float2(MMA_OP_SCALE, MMA_OP_SCALE)) {
        if constexpr (F16) {
            split_f16(fmul2(v, scale), hi[2 * b + h], lo[2 * b + h]);
        } else {
            split_tf32(v.x, hi[h], lo[h]);
            split_tf32(v.y, hi[2 + h], lo[2 + h]);
        }
    };
    auto mma = [&](float (&acc)[4], const unsigned (&x)[4], unsigned w0, unsigned w1) {
        if constexpr (F16) {
            mma_f16(acc, x, w0, w1);
        } else {
            const unsigned w[2] = {w0, w1};
            mma_tf32(acc, x, w, acc);
        }
    };
    for (int i = tid; i < N; i += C::THREADS) {
        sb[i] = i < n ? hd.b_h[i] + (proj ? hd.b_i[i] : 0.0f) : 0.0f;
        sb[N + i] = i < n ? hd.b_h[n + i] + (proj ? hd.b_i[n + i] : 0.0f) : 0.0f;
        sb[2 * N + i] = i < n ? hd.b_h[2 * n + i] : 0.0f;
        sb[3 * N + i] = i < n && proj ? hd.b_i[2 * n + i] : 0.0f;
    }
    const long long k0 = (long long)blockIdx.x * NC;
    const int nk = (int)min((long long)NC, total - k0);
    for (int k = tid; k < C::NC_MAX; k += C::THREADS) {
        SegChain ch{0, 0, 0, 0, 0};
        if (k < nk) {
            const long long q = (k0 + k) / nchain, b = q / s;
            const int c = (int)(k0 + k - q * nchain), ph = (int)(q - b * s), len = (a.T - ph + s - 1) / s;
            ch.e = b * a.T + ph;
            ch.b = (int)b;
            ch.t0 = c * L;
            ch.t_end = c * L < len ? min(len, (c + 1) * L) : 0;
            ch.next = (c + 1) * L < len;
        }
        tab[k] = ch;
    }
    pdl_prologue();
    if (*(volatile int *)&st->done) return;
    __syncthreads();
    const bool has_next = nk == NC && tab[NC - 1].next, has_prev = tab[0].t0 > 0 && tab[0].t_end > 0;
    const int G = NC >> 4;                               // groups (a power of two)

    int iters = *(volatile int *)&st->iters, burn = min(*(volatile int *)&st->burn, a.burn_cap), need = 0;       // (the slots end there)
    const float tol = st->tol;
    const int max_iter = st->max_iter;
    __shared__ unsigned red[4][C::WARPS];
    unsigned long long *const edge_w = reinterpret_cast<unsigned long long *>(a.edge) + (size_t)hd.first_edge * n;

    for (unsigned round = 1;; ++round) {
    const float *ycur = a.buf[iters & 1];
    float *ynew = a.buf[(iters + 1) & 1];
    const bool zero = iters == 0 && !a.warm;
    unsigned mb = 0u, mis = 0u;
    const bool xv2 = (m & 1) == 0 && ((uintptr_t)a.x & 7) == 0;
    auto ld2 = [&](const float *p, int col, int width) -> float2 {
        if constexpr (V2) {
            return col < width ? __ldcg(reinterpret_cast<const float2 *>(p + col)) : make_float2(0.0f, 0.0f);
        } else {
            return make_float2(col < width ? __ldcg(p + col) : 0.0f, col + 1 < width ? __ldcg(p + col + 1) : 0.0f);
        }
    };
    auto ldx = [&](const float *p, int col) -> float2 {
        if (xv2) return col < m ? __ldg(reinterpret_cast<const float2 *>(p + col)) : make_float2(0.0f, 0.0f);
        return make_float2(col < m ? __ldg(p + col) : 0.0f, col + 1 < m ? __ldg(p + col + 1) : 0.0f);
    };

    // ---------------------------------------------------------------- phase 1: the cell at every slot
    // A tile is one position of each of the sixteen chains of a group (warp w: group w % G, positions w / G, + WARPS / G, ...),
    // then sixteen consecutive positions of the first chain's burn-in.  Rows advance by constant strides; the next tile's
    // iterate is requested before the current one is used.
    const int burn0 = tab[0].t_end > 0 ? min(burn, tab[0].t0) : 0;       // positions of that burn-in
    const long long yst = (long long)s * H * n, xst = (long long)s * (proj ? m : H * 3 * n);
    for (int part = 0; part < 2; ++part) {
    const int dt = part == 0 ? C::WARPS / G : 16 * C::WARPS;             // positions between a row's tiles
    int left, tp[2], tlim[2], slot[2];
    const float *yp[2], *xp[2], *y0p[2];
    {
        const int first = part == 0 ? warp / G : (C::WARPS - 1 - warp) * 16;      // (the warps with fewest tiles of part 0)
        left = part == 0 ? (L - first + dt - 1) / dt : (burn0 - first + dt - 1) / dt;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = part == 0 ? (warp & (G - 1)) * 16 + g + 8 * h : 0;
            const SegChain ch = tab[k];
            tp[h] = part == 0 ? ch.t0 + first : ch.t0 - burn0 + first + g + 8 * h;
            tlim[h] = part == 0 ? ch.t_end : ch.t0;
            slot[h] = part == 0 ? burn + k * L + first : burn - burn0 + first + g + 8 * h;
            const long long e = ch.e + (long long)tp[h] * s;
            yp[h] = ycur + (e * H + blockIdx.y) * n;
            xp[h] = proj ? a.x + e * m : a.u + (e * H + blockIdx.y) * 3 * n;
            y0p[h] = a.y0 + ((long long)ch.b * H + blockIdx.y) * n;
        }
    }
    float nhp[NT][4], ny4[NT][4];
    float2 nx[2 * KB];
    auto fetch = [&]() {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const bool in = tp[h] < tlim[h], lh = in && (!zero || tp[h] == 0), ly = in && !zero;
            const float *hq = tp[h] == 0 ? y0p[h] : yp[h] - yst;
            if (proj) {
#pragma unroll
                for (int b = 0; b < KB; ++b) nx[2 * b + h] = in ? ldx(xp[h], 8 * b + 2 * t) : make_float2(0.0f, 0.0f);
            }
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                const float2 v = lh ? ld2(hq, 8 * j + 2 * t, n) : make_float2(0.0f, 0.0f);
                const float2 v2 = ly ? ld2(yp[h], 8 * j + 2 * t, n) : make_float2(0.0f, 0.0f);
                nhp[j][2 * h] = v.x; nhp[j][2 * h + 1] = v.y;
                ny4[j][2 * h] = v2.x; ny4[j][2 * h + 1] = v2.y;
            }
        }
    };
    if (left > 0) fetch();
    for (; left > 0; --left) {
        float hp[NT][4], y4[NT][4];
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) { hp[j][q] = nhp[j][q]; y4[j][q] = ny4[j][q]; }
        const bool act[2] = {tp[0] < tlim[0], tp[1] < tlim[1]};
        const float *xpp[2] = {xp[0], xp[1]};
        float *const so[2] = {slots + slot[0] * SZ, slots + slot[1] * SZ};
        const bool hid = __any_sync(0xffffffffu, !zero || tp[0] == 0 || tp[1] == 0);
#pragma unroll
        for (int h = 0; h < 2; ++h) { tp[h] += dt; slot[h] += dt; yp[h] += dt * yst; xp[h] += dt * xst; }
        float xr[NT][4], xz[NT][4], xn[NT][4];
        if (proj) {
            float2 xc[2 * KB];
#pragma unroll
            for (int q = 0; q < 2 * KB; ++q) xc[q] = nx[q];
            if (left > 1) fetch();
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int q = 0; q < 4; ++q) { xr[j][q] = 0.0f; xz[j][q] = 0.0f; xn[j][q] = 0.0f; }
#pragma unroll 1
            for (int kk = 0; kk < kx; ++kk) {
                unsigned ah[4], al[4];
#pragma unroll
                for (int q = 0; q < 2 * KB; ++q) operand(ah, al, q >> 1, q & 1, xc[q], *reinterpret_cast<const float2 *>(s_xf + (F16 ? 16 * kk + 8 * (q >> 1) + 2 * t : 0)));
                if (kk + 1 < kx) {
#pragma unroll
                    for (int q = 0; q < 2 * KB; ++q) xc[q] = act[q & 1] ? ldx(xpp[q & 1], 8 * KB * (kk + 1) + 8 * (q >> 1) + 2 * t) : make_float2(0.0f, 0.0f);
                }
                const uint4 *q0 = sI + (4 * kk + t) * NS + g;
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int gate = 0; gate < 3; ++gate) {
                        const uint4 w = q0[gate * N + 8 * j];
                        float (&acc)[4] = gate == 0 ? xr[j] : gate == 1 ? xz[j] : xn[j];
                        mma(acc, al, w.x, w.y);
                        mma(acc, ah, w.z, w.w);
                        mma(acc, ah, w.x, w.y);
                    }
            }
        } else {
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const int col = 8 * j + 2 * t;
                    const bool on = act[h] && col < n;
                    const float2 vr = on ? ld2(xpp[h], col, n) : make_float2(0.0f, 0.0f);
                    const float2 vz = on ? ld2(xpp[h] + n, col, n) : make_float2(0.0f, 0.0f);
                    const float2 vn = on ? ld2(xpp[h] + 2 * n, col, n) : make_float2(0.0f, 0.0f);
                    xr[j][2 * h] = vr.x; xr[j][2 * h + 1] = vr.y;
                    xz[j][2 * h] = vz.x; xz[j][2 * h + 1] = vz.y;
                    xn[j][2 * h] = vn.x; xn[j][2 * h + 1] = vn.y;
                }
            if (left > 1) fetch();
            if constexpr (F16) {                         // (in the products' scale: a power of two)
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int q = 0; q < 4; ++q) { xr[j][q] *= unit; xz[j][q] *= unit; xn[j][q] *= unit; }
            }
        }
        unsigned ah[NB][4], al[NB][4];
        if constexpr (F16 && NT % 2) {
#pragma unroll
            for (int q = 2; q < 4; ++q) { ah[NB - 1][q] = 0u; al[NB - 1][q] = 0u; }
        }
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) operand(ah[j / KB], al[j / KB], j % KB, h, make_float2(hp[j][2 * h], hp[j][2 * h + 1]));
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            {
                float (&hr)[4] = xr[j], (&hz)[4] = xz[j];
                float hq[4] = {0.f, 0.f, 0.f, 0.f};
                if (hid) {
                    const uint4 *q0 = sH + t * NS + 8 * j + g;
#pragma unroll
                    for (int kk = 0; kk < NB; ++kk)
#pragma unroll
                        for (int gate = 0; gate < 3; ++gate) {
                            const uint4 w = q0[4 * kk * NS + gate * N];
                            float (&acc)[4] = gate == 0 ? hr : gate == 1 ? hz : hq;
                            mma(acc, al[kk], w.x, w.y);
                            mma(acc, ah[kk], w.z, w.w);
                            mma(acc, ah[kk], w.x, w.y);
                        }
                }
                const int col = 8 * j + 2 * t;
                const float2 bR = *reinterpret_cast<const float2 *>(sb + col), bZ = *reinterpret_cast<const float2 *>(sb + N + col);
                const float2 bQ = *reinterpret_cast<const float2 *>(sb + 2 * N + col), bN = *reinterpret_cast<const float2 *>(sb + 3 * N + col);
                const float2 one = make_float2(1.0f, 1.0f), mone = make_float2(-1.0f, -1.0f), k2 = make_float2(kS, kS);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float2 y2 = make_float2(y4[j][2 * h], y4[j][2 * h + 1]);
                    const float2 h2 = make_float2(hp[j][2 * h], hp[j][2 * h + 1]);
                    const float2 q = ffma2(make_float2(hq[2 * h], hq[2 * h + 1]), k2, bQ);
                    const float2 r = sigmoid2_gate(ffma2(make_float2(hr[2 * h], hr[2 * h + 1]), k2, bR));
                    const float2 z = sigmoid2_gate(ffma2(make_float2(hz[2 * h], hz[2 * h + 1]), k2, bZ));
                    const float2 c = tanh2_gate(ffma2(r, q, ffma2(make_float2(xn[j][2 * h], xn[j][2 * h + 1]), k2, bN)));
                    const float2 omz = ffma2(z, mone, one), omr = ffma2(r, mone, one);
                    const float2 f = ffma2(omz, c, fmul2(z, h2));
                    // (the three coefficients of products with the update carry their scale)
                    const float2 kd = make_float2(kD, kD), okd = F16 ? fmul2(omz, kd) : omz;
                    const float2 az = fmul2(fmul2(ffma2(c, mone, h2), z), okd);
                    const float2 an = fmul2(okd, ffma2(fmul2(c, mone), c, one));
                    const float2 kn = fmul2(an, r);
                    const float2 kr = fmul2(fmul2(kn, q), omr);
                    if (act[h]) {
                        float *o = so[h] + col;
                        *reinterpret_cast<float2 *>(o) = z;
                        *reinterpret_cast<float2 *>(o + N) = kr;
                        *reinterpret_cast<float2 *>(o + 2 * N) = az;
                        *reinterpret_cast<float2 *>(o + 3 * N) = kn;
                        *reinterpret_cast<float2 *>(o + 4 * N) = ffma2(y2, mone, f);
                    }
                }
            }
        }
    }
    }
    __syncthreads();

    // ---------------------------------------------------------------- phase 2: the chains
    const int grp = warp / NT, j = warp % NT;            // this warp: columns 8j .. 8j + 7 of the chains of group grp
    const bool live = grp < G && grp * 16 < nk;
    float d[4] = {0.f, 0.f, 0.f, 0.f};
    bool next[2] = {false, false}, gave_up = false;
    if (live) {
        uint4 wf[N <= 32 ? NB : 1][3];
        const uint4 *wq = sH + t * NS + 8 * j + g;
        if constexpr (N <= 32) {
#pragma unroll
            for (int kk = 0; kk < NB; ++kk)
#pragma unroll
                for (int gate = 0; gate < 3; ++gate) wf[kk][gate] = wq[4 * kk * NS + gate * N];
        }
        int tt[2], t_end[2], t_own[2];
        const float *cf[2];
        float *yn[2];
        ptrdiff_t to_old = ycur - ynew;
        const size_t ys = (size_t)s * H * n;
        const int col = 8 * j + 2 * t;
        int lead = burn;                                 // no chain of the group has a burn-in: start behind it
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = grp * 16 + g + 8 * h;
            const SegChain ch = tab[k];
            tt[h] = ch.t0 - burn;
            t_end[h] = ch.t_end;
            t_own[h] = ch.t0;
            next[h] = ch.next != 0;
            cf[h] = slots + (size_t)(k < nk ? k : 0) * L * SZ + col;
            yn[h] = ynew + (((size_t)ch.e + (size_t)ch.t0 * s) * H + blockIdx.y) * n + col;
            if (ch.t_end > 0 && ch.t0 > 0) lead = max(0, min(lead, burn - ch.t0));
        }
        lead = __reduce_min_sync(0xffffffffu, lead);
        tt[0] += lead; tt[1] += lead;
        cf[0] += (size_t)lead * SZ; cf[1] += (size_t)lead * SZ;
        float *xrow = dx + (size_t)grp * 16 * DS;
        if constexpr (NT > 1) {                          // zero entering updates in the buffer the first step reads
            float *x0 = xrow;
            *reinterpret_cast<float2 *>(x0 + g * DS + col) = make_float2(0.f, 0.f);
            *reinterpret_cast<float2 *>(x0 + (g + 8) * DS + col) = make_float2(0.f, 0.f);
        }
        auto group_sync = [&]() {
            if constexpr (NT > 1) asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "r"(32 * NT) : "memory");
        };
        // one step: the coefficients of the next one are read while the products of this one run
        float2 cz[2], ckr[2], caz[2], ckn[2], cr[2];
        auto load_coefs = [&]() {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                cz[h] = *reinterpret_cast<const float2 *>(cf[h]);
                ckr[h] = *reinterpret_cast<const float2 *>(cf[h] + N);
                caz[h] = *reinterpret_cast<const float2 *>(cf[h] + 2 * N);
                ckn[h] = *reinterpret_cast<const float2 *>(cf[h] + 3 * N);
                cr[h] = *reinterpret_cast<const float2 *>(cf[h] + 4 * N);
                cf[h] += SZ;
            }
        };
        int buf = 0;
        auto advance = [&](bool more) {
            float u[3][4], v[3][4], w2[3][4];            // hi.hi, and the two cross terms beside it
#pragma unroll
            for (int gate = 0; gate < 3; ++gate)
#pragma unroll
                for (int q = 0; q < 4; ++q) { u[gate][q] = 0.f; v[gate][q] = 0.f; w2[gate][q] = 0.f; }
            const float *xin = xrow + buf * (C::NC_MAX * DS);
#pragma unroll
            for (int kk = 0; kk < NB; ++kk) {
                unsigned dh[4], dl[4];
                if constexpr (F16) {                     // (the pairs of columns are exchanged as the operand's halves)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (2 * kk + (q >> 1) < NT) {
                            const uint2 p = *reinterpret_cast<const uint2 *>(xin + (g + 8 * (q & 1)) * DS + 16 * kk + 8 * (q >> 1) + 2 * t);
                            dh[q] = p.x; dl[q] = p.y;
                        } else {
                            dh[q] = 0u; dl[q] = 0u;
                        }
                    }
                } else {
                    float2 p[2] = {make_float2(d[0], d[1]), make_float2(d[2], d[3])};
                    if constexpr (NT > 1) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) p[h] = *reinterpret_cast<const float2 *>(xin + (g + 8 * h) * DS + 8 * kk + 2 * t);
                    }
                    operand(dh, dl, 0, 0, p[0]);
                    operand(dh, dl, 0, 1, p[1]);
                }
#pragma unroll
                for (int gate = 0; gate < 3; ++gate) {
                    uint4 w;
                    if constexpr (N <= 32) w = wf[kk][gate]; else w = wq[4 * kk * NS + gate * N];
                    mma(u[gate], dh, w.x, w.y);
                    if constexpr (EXACT) {
                        mma(v[gate], dl, w.x, w.y);
                        mma(w2[gate], dh, w.z, w.w);
                    }
                }
            }
            buf ^= 1;
            float *xout = xrow + buf * (C::NC_MAX * DS);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool act = tt[h] >= 0 && tt[h] < t_end[h];
                const float2 d2 = make_float2(d[2 * h], d[2 * h + 1]);
                float2 o = ffma2(cz[h], d2, cr[h]);
                const float2 ck[3] = {ckr[h], caz[h], ckn[h]};
                if constexpr (EXACT) {
#pragma unroll
                    for (int gate = 0; gate < 3; ++gate)
                        o = ffma2(ck[gate], fadd2(make_float2(v[gate][2 * h], v[gate][2 * h + 1]), make_float2(w2[gate][2 * h], w2[gate][2 * h + 1])), o);
                }
#pragma unroll
                for (int gate = 0; gate < 3; ++gate) o = ffma2(ck[gate], make_float2(u[gate][2 * h], u[gate][2 * h + 1]), o);
                d[2 * h] = act ? o.x : d[2 * h];
                d[2 * h + 1] = act ? o.y : d[2 * h + 1];
                if constexpr (F16) {
                    uint2 p;
                    split_f16(fmul2(make_float2(d[2 * h], d[2 * h + 1]), make_float2(MMA_D_SCALE, MMA_D_SCALE)), p.x, p.y);
                    *reinterpret_cast<uint2 *>(xout + (g + 8 * h) * DS + col) = p;
                } else if constexpr (NT > 1) {
                    *reinterpret_cast<float2 *>(xout + (g + 8 * h) * DS + col) = make_float2(d[2 * h], d[2 * h + 1]);
                }
            }
            if (more) load_coefs();
            group_sync();
        };
        // the old iterate of its own positions is requested AHEAD steps before it is used (the first ones behind the burn-in)
        constexpr int AHEAD = 4;
        float2 yo[AHEAD][2];
        auto load_old = [&](int i, int off, float2 (&y2)[2]) {           // position i, `off` positions ahead of yn
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                y2[h] = make_float2(0.f, 0.f);
                if (!zero && i < L && t_own[h] + i < t_end[h]) y2[h] = ld2(yn[h] - col + to_old + (size_t)off * ys, col, n);
            }
        };
#pragma unroll
        for (int q = 0; q < AHEAD; ++q) load_old(q, q, yo[q]);
        group_sync();
        load_coefs();
#pragma unroll 1
        for (int step = lead; step < burn; ++step) {
            advance(true);
            ++tt[0]; ++tt[1];
        }
        *reinterpret_cast<float2 *>(ss + (grp * 16 + g) * DS + col) = make_float2(d[0], d[1]);
        *reinterpret_cast<float2 *>(ss + (grp * 16 + g + 8) * DS + col) = make_float2(d[2], d[3]);
        if (whole_loop && has_prev && grp == 0 && g == 0) {              // the start state this CTA's first chain assumed
            st_word(edge_w + (size_t)blockIdx.x * n, col, n, d[0], round);
            st_word(edge_w + (size_t)blockIdx.x * n, col + 1, n, d[1], round);
        }
#pragma unroll 1
        for (int i0 = 0; i0 < L; i0 += AHEAD) {
#pragma unroll
            for (int q = 0; q < AHEAD; ++q) {
                const int i = i0 + q;
                if (i < L) {
                    advance(i + 1 < L);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (tt[h] < t_end[h]) {
                            const float2 old = yo[q][h], yv = make_float2(old.x + d[2 * h], old.y + d[2 * h + 1]);
                            if (col < n) mb = max(mb, absdiff_bits(yv.x, old.x));
                            if (col + 1 < n) mb = max(mb, absdiff_bits(yv.y, old.y));
                            if constexpr (V2) { if (col < n) *reinterpret_cast<float2 *>(yn[h]) = yv; }
                            else { if (col < n) yn[h][0] = yv.x; if (col + 1 < n) yn[h][1] = yv.y; }
                        }
                        ++tt[h];
                        yn[h] += ys;
                    }
                    load_old(i + AHEAD, AHEAD - 1, yo[q]);
                }
            }
        }
        // the boundary behind this CTA: its successor's assumed start was posted when that one's burn-in ended
        if (whole_loop && has_next && grp == G - 1 && g == 7) {
            const unsigned long long *q = edge_w + (size_t)(blockIdx.x + 1) * n + col;
            if (col < n) mis = max(mis, absdiff_bits(d[2], __uint_as_float(wait_word(q, round, gave_up))));
            if (col + 1 < n) mis = max(mis, absdiff_bits(d[3], __uint_as_float(wait_word(q + 1, round, gave_up))));
        }
    }
    __syncthreads();
    // ---------------------------------------------------------------- boundaries
    float *send = dx;                                    // end state of the last chain (the exchange buffers are free)
    if (live) {
        const int col = 8 * j + 2 * t;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = grp * 16 + g + 8 * h;
            if (next[h] && k + 1 < nk) {
                const float2 v = *reinterpret_cast<const float2 *>(ss + (k + 1) * DS + col);
                mis = max(mis, max(absdiff_bits(v.x, d[2 * h]), absdiff_bits(v.y, d[2 * h + 1])));
            }
            if (k == NC - 1) *reinterpret_cast<float2 *>(send + col) = make_float2(d[2 * h], d[2 * h + 1]);
        }
    }
    __syncthreads();
    if (whole_loop) {
        // The CTAs of a cooperative launch are all resident, so they may wait for one another.  The successor's assumed start
        // was posted when its burn-in ended; then every CTA posts its two maxima and reads everybody's: one exchange through
        // L2 is both the barrier and the reduction, and the decision is taken by all CTAs alike.
        mb = __reduce_max_sync(0xffffffffu, mb);
        mis = __reduce_max_sync(0xffffffffu, mis);
        if (lane == 0) { red[0][warp] = mb; red[1][warp] = mis; }
        __syncthreads();
        unsigned long long *box = a.words + ((size_t)blockIdx.y * 2 + (round & 1)) * 2 * gridDim.x;
        if (warp == 0) {
            const unsigned e = __reduce_max_sync(0xffffffffu, lane < C::WARPS ? red[0][lane] : 0u);
            const unsigned q = __reduce_max_sync(0xffffffffu, lane < C::WARPS ? red[1][lane] : 0u);
            if (lane == 0 && !(a.expire && blockIdx.x == 0)) {             // (expire: nobody's wait for the first CTA ends)
                __threadfence();                         // this CTA's part of the new iterate is visible before its word
                st_relaxed_u64w(box + 2 * blockIdx.x, ((unsigned long long)round << 32) | e);
                st_relaxed_u64w(box + 2 * blockIdx.x + 1, ((unsigned long long)round << 32) | q);
            }
        }
        unsigned e = 0u, q = 0u;
        for (int i = tid; i < (int)nctas; i += C::THREADS) {
            e = max(e, wait_word(box + 2 * i, round, gave_up));
            if (!gave_up) q = max(q, wait_word(box + 2 * i + 1, round, gave_up));
        }
        e = __reduce_max_sync(0xffffffffu, e);
        q = __reduce_max_sync(0xffffffffu, q);
        if (lane == 0) { red[2][warp] = e; red[3][warp] = q; }
        if (__syncthreads_or(gave_up)) {                 // a bounded wait ran out: every CTA drains the same way
            if (tid == 0) { atomicOr(&st->flags, FLAG_TIMEOUT); st->done = BODY_DONE; }
            return;
        }
        const unsigned eb = __reduce_max_sync(0xffffffffu, lane < C::WARPS ? red[2][lane] : 0u);
        const unsigned qb = __reduce_max_sync(0xffffffffu, lane < C::WARPS ? red[3][lane] : 0u);
        BodyVerdict v = body_verdict(__uint_as_float(eb), __uint_as_float(qb), a.eta, burn, a.burn_cap, a.T, tol, iters, max_iter, a.adapt != 0, 0.0f);
        if (F16 && (!(__uint_as_float(eb) <= 3.402823466e38f) || !(__uint_as_float(qb) <= 3.402823466e38f)))
            v = BodyVerdict{false, BODY_BEYOND, 0, 0};
        need = max(need, v.need);
        if (blockIdx.x == 0 && tid == 0) {
            if (v.counts) {
                if (st->trace && iters < ERR_TRACE_CAP) st->trace[iters] = __uint_as_float(eb);
                if (st->host && iters < HOST_TRACE) st->host->trace[iters] = __uint_as_float(eb);
                st->err_last_bits = eb;
            }
            if (v.done) {
                st->iters = iters + (v.counts ? 1 : 0);
                const int told = v.done == BODY_DONE ? need : v.burn;
                st->burn = told;
                st->done = v.done;
                if (HostResult *h = st->host) post_result(h, v.done, told, st->iters, st->err_last_bits, a.polled || v.done != BODY_DONE);
            }
        }
        if (v.done) return;
        iters += v.counts ? 1 : 0;
        burn = v.burn;
        continue;
    }
    if (warp < 2 && (warp == 0 ? has_next : has_prev)) { // warp 0: the boundary behind this CTA, warp 1: the one before it
        const int side = warp;
        const size_t edge = (size_t)hd.first_edge + blockIdx.x - side;
        const float *own = side == 0 ? send : ss;
        float *slot = a.edge + edge * 2 * n;
        for (int i = lane; i < n; i += 32) __stcg(slot + side * n + i, own[i]);
        __threadfence();
        __syncwarp();
        unsigned old = 0;
        if (lane == 0) old = atomicAdd(a.edge_flag + edge, 1u);
        old = __shfl_sync(0xffffffffu, old, 0);
        if (old == 1u) {
            __threadfence();
            for (int i = lane; i < n; i += 32) mis = max(mis, absdiff_bits(own[i], __ldcg(slot + (side ^ 1) * n + i)));
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
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        const unsigned prev = atomicAdd(&st->exit_counter, 1u);
        if (prev + 1u == nctas) {
            __threadfence();
            st->exit_counter = 0u;
            body_decide(st, a, 1, 0.0f, F16);
        }
    }
    return;
    }
}

}  // namespace deer
