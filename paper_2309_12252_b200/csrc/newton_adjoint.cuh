// The gradient's adjoint solve as ONE launch (Eq. 7; the dual operator of Sec. 3.1.1): gates at the trajectory,
// lambda_t = gy_t + J_{t+1}^T lambda_{t+1}, and the gradients w.r.t. the pre-activations -- no projected inputs, Jacobians,
// coefficient rows or lambda in memory.
//
// Chains in lockstep, burn-in and verified boundaries as in newton_body.cuh, in descending time.  The state that a chain
// carries is mu_t = J_{t+1}^T lambda_{t+1}.  With the gates at t and lambda = gy + mu, the hidden-side gradients of the three
// pre-activations are p = (k_r.lambda, a_z.lambda, k_n.lambda) -- what dW_h, dW_i, dx are contractions of -- and
//     J_t^T lambda = z.lambda + p W_h        [16, 3n] x [3n, n], p's accumulator layout being the A operand as it stands
//                                            (a pair of blocks of eight columns is one K step of 16).
// All products are at fp32 level (a one-shot solve): three TF32 MMAs on split operands up to n = 16, from there on hi + lo f16
// halves in three m16n8k16 ones, half as many and good to 2^-22 of the operands (small ones to 2^-27 of a state and of what x
// contributes to a gate, 2^-34 of the row's largest |lambda|) where those are to 2^-20.  Powers of two (operand_scales, and per row
// and step one from the row's largest |lambda|) keep the halves among the normal numbers; a value beyond f16's range makes a NaN,
// which fails the check below.  lambda has no scale that holds everywhere: a sequence's loss may weigh a millionth of another's, and behind a loss on the last step only lambda decays through every magnitude, down to dx and dy0 at
// the first one.  So a boundary is held to eta of the largest |lambda| of all and, besides, to ADJ_LOCAL eta of the largest
// |lambda| just before it, over the last ADJ_WINDOW positions of its successor's burn-in (one position alone may be near zero
// where n is small; more would measure a decayed lambda by what it decayed from).  Where all losses weigh alike the window's
// largest is some third of the largest of all, so that the first rule decides there.
// One boundary that differs by more leaves StatusBlock::done at 0: the launches enqueued behind this one (a longer burn-in,
// then the kernels that multiply the Jacobians out) do the work.
// What bounds it: the latency of chained mma.sync with eight warps per SM (254 registers a thread).  n = m = 32, B = 16, T = 2e4: tensor
// pipe 34 % active, issue slots 32 % used, DRAM 17 % (in TF32 48, 32 and 15 %, and 506 us under the profiler where it now takes 396);
// T = 1e5 takes 820 us where it took 1100.
// The boundaries that dy0 can still feel -- those less than DY0_REACH burn-ins from the sequence's first step -- are held to
// eta * max|dy0| as well.
#pragma once
#include "newton_body.cuh"

namespace deer {

constexpr int DY0_REACH = 8;     // a burn-in takes an error down by about 1e-6 or more; behind eight of them it is below any fp32
constexpr int ADJ_WINDOW = 8;    // positions before a boundary whose largest |lambda| is its scale
constexpr float ADJ_LOCAL = 4.0f;
constexpr int ADJ_TOP = 12;      // of a channel's largest weight (operand_scales): contributions up to 16,376, held to 2^-27 absolute.  There is no
                                 // second try with projected inputs here, as an evaluation has it
static_assert(ADJ_WINDOW <= ADJ_BURN && (ADJ_BURN - ADJ_WINDOW) % 4 == 0, "the window is whole steps of every kernel's burn-in");

// A boundary's mismatch as a part of its scale, as the bits of a non-negative float (a NaN stays above all numbers).
__device__ __forceinline__ unsigned boundary_ratio(unsigned diff, float scale)
{
    return diff == 0u ? 0u : __float_as_uint(fabsf(__uint_as_float(diff) / scale));
}

template <int N> struct Adj {
    static constexpr int NT = N / 8;
    // f16 halves from n = 17 on.  Up to 16 the products are few: their halves' conversions and p's scale, which is in the chain, cost
    // what half the MMAs give.  (us per gradient, TF32 / f16: n = 16, m = 4, 1.28e6 positions 698 / 720; 30 heads of 16 1486 / 1520,
    // 32 of 8 2147 / 2191; n = 24, m = 16, 1.6e5 390 / 386; n = m = 32 520 / 448; n = 48, m = 32, 64,000 957 / 660; n = 56, m = 8,
    // 48,000 1100 / 760.)
    static constexpr bool F16 = NT > 2;
    static constexpr int KB = F16 ? 2 : 1;               // column blocks of a K step
    static constexpr int NB = (NT + KB - 1) / KB, PB = (3 * NT + KB - 1) / KB;       // K steps of h and of p
    static constexpr int NS = 3 * N + 2, NS2 = N + 2;    // = 2 (mod 8) records
    static constexpr int SW = N + 4;
    static constexpr bool SS_GLOBAL = N > 48;            // start states in the workspace: the weights of both contractions fill
                                                         // the shared memory
    static constexpr size_t smem(int warps, int kx)
    {
        if (SS_GLOBAL) warps = 0;
        return sizeof(float) * ((size_t)16 * (NB + (kx + KB - 1) / KB) * NS + (size_t)16 * PB * NS2 + 4 * N + (size_t)warps * 16 * SW);
    }
};

// The burn-in of this launch: the call's, or what the launch before this one found to be needed (0: more than is worth trying).
__device__ __forceinline__ int adjoint_burn(const AdjArgs &a, const StatusBlock *st)
{
    const int want = *(const volatile int *)&st->burn;
    return want == 0 ? a.burn : want <= a.burn_cap ? want : 0;
}

// End of the launch: were the boundaries good enough?  Single thread.
__device__ __forceinline__ void adjoint_decide(StatusBlock *st, float eta, bool dy0, int burn)
{
    // (all words are requested before the first is looked at)
    const unsigned flags = *(volatile unsigned *)&st->flags;
    auto word = [](unsigned &w) { return __uint_as_float(*(volatile unsigned *)&w); };
    const float top = word(st->err_bits), mis = word(st->mis_bits), rel = word(st->rel_bits), top_end = word(st->top_end_bits), mis_end = word(st->mis_end_bits);
    st->err_bits = 0u; st->mis_bits = 0u; st->rel_bits = 0u; st->top_end_bits = 0u; st->mis_end_bits = 0u;
    if (flags & FLAG_TIMEOUT) { st->burn = 1 << 20; return; }            // (unfinished rows: the kernels behind do the work)
    // (at the first time step a NaN reaches no boundary and no lambda any more, only the final state and the gradients there)
    const bool inner = top_end <= 3.402823466e38f && mis <= eta * top && rel <= ADJ_LOCAL * eta, end = !dy0 || mis_end <= eta * top_end;
    if (inner && end) { st->done = BODY_DONE; return; }
    // the carried error is about |lambda| * rho^burn: the burn-in after which it is half of what is accepted
    int want = 1 << 20;
    if (inner) want = 3 * burn;
    else if (mis < 0.7f * top && rel < 0.7f) want = (int)(1.1f * (float)burn * __logf(0.5f * eta) / __logf(fmaxf(mis / top, rel / ADJ_LOCAL))) + 4;
    st->burn = max(want, burn + 8);
}

// CTAS: per SM, at n = 9 to 16 two, which need not spill, or three where many channels are contracted, which leave a step with too
// little to do beside it.  (us per gradient, three / two: n = 16, m = 8, 240,000 positions 300 / 252, 960,000 572 / 560; m = 24,
// 640,000 534 / 500; m = 64, 640,000 780 / 922; n = 12, m = 8, 320,000 435 / 396, m = 40 650 / 605; 31 heads of 16 1955 / 1915.)
template <int N> __host__ __device__ constexpr int adjoint_ctas(int m) { return N > 32 ? 1 : N > 16 ? 2 : N > 8 ? (m > 40 ? 3 : 2) : 3; }

template <int N, bool V2, int CTAS>
__global__ void __launch_bounds__(N > 32 ? 256 : 128, CTAS) newton_adjoint_kernel(AdjArgs a)
{
    using C = Adj<N>;
    constexpr int NT = C::NT, KB = C::KB, NB = C::NB, PB = C::PB, NS = C::NS, NS2 = C::NS2, SW = C::SW;
    constexpr bool F16 = C::F16;
    extern __shared__ __align__(16) float smb[];
    __shared__ unsigned s_top;
    __shared__ __align__(16) float s_xf[64];
    const BodyHead hd = a.heads ? a.heads[blockIdx.y] : a.h0;
    StatusBlock *st = a.st + blockIdx.y;
    const int n = a.n, m = a.m, H = a.H, L = a.L;
    const bool proj = a.u == nullptr;
    const int kx = proj ? (m + 8 * KB - 1) / (8 * KB) : 0;               // K steps of x
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int g = lane >> 2, t = lane & 3;

    // geometry of this CTA's head
    const int s = hd.stride, Tp = (a.T + s - 1) / s, nchain = (Tp + L - 1) / L;
    const long long total = (long long)a.B * s * nchain;
    const long long groups = (total + 15) >> 4;
    const unsigned nctas = (unsigned)((groups + nwarps - 1) / nwarps);
    if (blockIdx.x >= nctas) return;

    // ---- weights into shared memory as records of the four words that a lane needs for a column of a K step: hi of rows 2t, 2t + 1
    // (and 2t + 8, 2t + 9), and lo of the same: one 128-bit load (weights are not produced by the previous launch: this runs
    // before its end)
    uint4 *sH = reinterpret_cast<uint4 *>(smb), *sI = sH + 4 * NB * NS;
    uint4 *sT = sI + 4 * kx * NS;                        // W_h by rows: the B operand of p W_h
    float *sb = reinterpret_cast<float *>(sT + 4 * PB * NS2);
    float wscale = 1.0f, unit = 1.0f, kS = 1.0f;
    if constexpr (F16) {
        wscale = operand_scales(hd.W_h, hd.W_i, 3 * n, n, proj ? m : 0, MMA_OP_SCALE, ADJ_TOP, s_xf, &s_top);
        unit = wscale * MMA_OP_SCALE;
        kS = 1.0f / unit;
    }
    auto record = [&](auto w, int kt) {                  // w(k): row k of the column
        const int k = 8 * KB * (kt >> 2) + 2 * (kt & 3);
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
    for (int idx = tid; idx < 4 * NB * 3 * N; idx += blockDim.x) {
        const int kt = idx % (4 * NB), c = idx / (4 * NB), gate = c / N, i = c % N;
        const float *wr = hd.W_h + (size_t)(gate * n + i) * n;
        sH[kt * NS + c] = record([&](int j) { return i < n && j < n ? wr[j] * wscale : 0.0f; }, kt);
    }
    for (int idx = tid; idx < 4 * kx * 3 * N; idx += blockDim.x) {
        const int kt = idx % (4 * kx), c = idx / (4 * kx), gate = c / N, i = c % N;
        const float *wr = hd.W_i + (size_t)(gate * n + i) * m;
        sI[kt * NS + c] = record([&](int j) { return i < n && j < m ? wr[j] * (F16 ? unit * pow2_inverse(s_xf[j]) : 1.0f) : 0.0f; }, kt);
    }
    for (int idx = tid; idx < 4 * PB * N; idx += blockDim.x) {
        const int c = idx % N, kt = idx / N;
        sT[kt * NS2 + c] = record([&](int j) { return j < 3 * N && j % N < n && c < n ? hd.W_h[(size_t)(j / N * n + j % N) * n + c] * wscale : 0.0f; }, kt);
    }
    for (int i = tid; i < N; i += blockDim.x) {          // (u holds b_i already)
        sb[i] = i < n ? hd.b_h[i] + (proj ? hd.b_i[i] : 0.0f) : 0.0f;
        sb[N + i] = i < n ? hd.b_h[n + i] + (proj ? hd.b_i[n + i] : 0.0f) : 0.0f;
        sb[2 * N + i] = i < n ? hd.b_h[2 * n + i] : 0.0f;
        sb[3 * N + i] = i < n && proj ? hd.b_i[2 * n + i] : 0.0f;
    }
    float *ss = sb + 4 * N + warp * 16 * SW;             // start states of this warp's chains
    if constexpr (C::SS_GLOBAL) ss = a.starts + ((size_t)hd.first_edge + (size_t)blockIdx.x * nwarps + warp) * 16 * SW;
    pdl_prologue();
    const int burn = adjoint_burn(a, st);
    if (*(volatile int *)&st->done || burn == 0) return;
    __syncthreads();

    const long long grp = (long long)blockIdx.x * nwarps + warp;
    unsigned mb = 0u, mis = 0u, rel = 0u, mb_end = 0u, mis_end = 0u;
    unsigned top[2] = {0u, 0u};                          // largest |mu| of this lane's columns of its two rows over the window

    if (grp < groups) {
        // ---- rows g and g + 8 of this lane: chain c of sequence (b, phase); scan position q is time step len - 1 - q
        int tt[2], t_end[2], len[2];
        const float *yp[2], *xp[2], *gp[2], *y0p[2];     // pointers at scan position tt (not dereferenced outside the sequence)
        long long row[2];                                // row of the scan position in [B,T]
        bool next[2];
        const long long ys = (long long)s * H * n, xs = (long long)s * (proj ? m : H * 3 * n);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const long long gid = grp * 16 + g + 8 * h;
            const long long q = gid < total ? gid / nchain : 0;
            const int c = gid < total ? (int)(gid - q * nchain) : 0;
            const long long b = q / s;
            const int ph = (int)(q - b * s);
            len[h] = gid < total ? (a.T - ph + s - 1) / s : 0;
            t_end[h] = min(len[h], (c + 1) * L);
            if (c * L >= len[h]) t_end[h] = 0;
            next[h] = (c + 1) * L < len[h];
            tt[h] = c * L - burn;
            const long long e = b * a.T + ph + (long long)(len[h] - 1 - tt[h]) * s;
            row[h] = e;
            yp[h] = a.y + (e * H + blockIdx.y) * n;
            gp[h] = a.gy + (e * H + blockIdx.y) * n;
            xp[h] = proj ? a.x + e * m : a.u + (e * H + blockIdx.y) * 3 * n;
            y0p[h] = a.y0 + ((size_t)b * H + blockIdx.y) * n;
        }
        // boundaries behind rows g, g + 8 and the one before row 0: close enough to the first time step for dy0 to feel them
        const int reach = DY0_REACH * burn;
        const bool near[2] = {len[0] - t_end[0] < reach, len[1] - t_end[1] < reach};
        const bool near_prev = __shfl_sync(0xffffffffu, (int)(len[0] - (tt[0] + burn) < reach), 0) != 0;
        // (a warp whose chains are all first ones has no burn-in: its earliest position is -burn)
        const int tmax = __reduce_max_sync(0xffffffffu, max(t_end[0] > 0 ? tt[0] : -burn, t_end[1] > 0 ? tt[1] : -burn));
        const int s_first = tmax <= -burn ? burn : 0;
        const int s_end = __reduce_max_sync(0xffffffffu, max(t_end[0] > 0 ? t_end[0] - tt[0] : 0, t_end[1] > 0 ? t_end[1] - tt[1] : 0));
#pragma unroll
        for (int h = 0; h < 2; ++h) { tt[h] += s_first; row[h] -= (long long)s_first * s; yp[h] -= s_first * ys; gp[h] -= s_first * ys; xp[h] -= s_first * xs; }

        auto ld2 = [&](const float *p, int col, int width) -> float2 {
            if constexpr (V2) {
                return col < width ? *reinterpret_cast<const float2 *>(p + col) : make_float2(0.0f, 0.0f);
            } else {
                return make_float2(col < width ? p[col] : 0.0f, col + 1 < width ? p[col + 1] : 0.0f);
            }
        };
        const bool xv2 = (m & 1) == 0 && ((uintptr_t)a.x & 7) == 0;
        auto ldx = [&](const float *p, int col) -> float2 {
            if (xv2) return col < m ? __ldg(reinterpret_cast<const float2 *>(p + col)) : make_float2(0.0f, 0.0f);
            return make_float2(col < m ? __ldg(p + col) : 0.0f, col + 1 < m ? __ldg(p + col + 1) : 0.0f);
        };
        // at scan position tt: the state before it (y0 before the first time step), dL/dy
        auto load_h = [&](float (&dst)[NT][4]) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool in = tt[h] >= 0 && tt[h] < t_end[h];
                const float *p = tt[h] == len[h] - 1 ? y0p[h] : yp[h] - ys;
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const float2 v = in ? ld2(p, 8 * j + 2 * t, n) : make_float2(0.0f, 0.0f);
                    dst[j][2 * h] = v.x; dst[j][2 * h + 1] = v.y;
                }
            }
        };
        auto load_g = [&](float (&dst)[NT][4]) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool in = tt[h] >= 0 && tt[h] < t_end[h];
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const float2 v = in ? ld2(gp[h], 8 * j + 2 * t, n) : make_float2(0.0f, 0.0f);
                    dst[j][2 * h] = v.x; dst[j][2 * h + 1] = v.y;
                }
            }
        };
        float hp[NT][4], gy[NT][4], d[NT][4];            // d: mu
        load_h(hp);
        load_g(gy);
#pragma unroll
        for (int j = 0; j < NT; ++j) { d[j][0] = d[j][1] = d[j][2] = d[j][3] = 0.0f; }

        // projected inputs at position tt + ahead
        constexpr bool U_AHEAD = NT <= 2;                // a step ahead where the registers allow it
        auto load_u = [&](float (&vr)[NT][4], float (&vz)[NT][4], float (&vn)[NT][4], int ahead) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool on = tt[h] + ahead >= 0 && tt[h] + ahead < t_end[h];
                const float *q = xp[h] - ahead * (ptrdiff_t)xs;
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const int col = 8 * j + 2 * t;
                    const float2 a0 = on ? ld2(q, col, n) : make_float2(0.0f, 0.0f);
                    const float2 a1 = on && col < n ? ld2(q + n, col, n) : make_float2(0.0f, 0.0f);
                    const float2 a2 = on && col < n ? ld2(q + 2 * n, col, n) : make_float2(0.0f, 0.0f);
                    vr[j][2 * h] = a0.x; vr[j][2 * h + 1] = a0.y;
                    vz[j][2 * h] = a1.x; vz[j][2 * h + 1] = a1.y;
                    vn[j][2 * h] = a2.x; vn[j][2 * h + 1] = a2.y;
                }
            }
        };
        float ur_n[U_AHEAD ? NT : 1][4], uz_n[U_AHEAD ? NT : 1][4], un_n[U_AHEAD ? NT : 1][4];
        if constexpr (U_AHEAD) { if (!proj) load_u(ur_n, uz_n, un_n, 0); }

        // block b of a K step of an A operand, row h of this lane: two columns (an accumulator's columns of TF32 in the slots t, t + 4)
        auto operand = [&](unsigned (&hi)[4], unsigned (&lo)[4], int b, int h, float2 v, float2 scale) {
            if constexpr (F16) {
                split_f16(fmul2(v, scale), hi[2 * b + h], lo[2 * b + h]);
            } else {
                split_tf32(v.x, hi[h], lo[h]);
                split_tf32(v.y, hi[2 + h], lo[2 + h]);
            }
        };
        // the lo halves: of TF32 formed where they are used (kept, they spill at n = 16: 1.28e6 positions 562 -> 580 us)
        auto low = [&](const unsigned (&hi)[4], unsigned (&lo)[4]) {
            if constexpr (!F16) {
#pragma unroll
                for (int q = 0; q < 4; ++q) { unsigned h; split_tf32(__uint_as_float(hi[q]), h, lo[q]); }
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

#pragma unroll 1
        for (int step = s_first; step < s_end; ++step) {
            // (mu stands for lambda = gy + mu in the window: work for eight steps instead of for every one, under the branch that the
            // burn-in's end has anyway; n = 33, 4,700 positions: 508 us without the scale, 514 so, 523 with a branch of its own)
            if (step > burn - ADJ_WINDOW && step <= burn) {
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int q = 0; q < 4; ++q) top[q >> 1] = max(top[q >> 1], __float_as_uint(fabsf(d[j][q])));
                if (step == burn) {                          // start states, and the scales of the boundaries before them
#pragma unroll
                    for (int j = 0; j < NT; ++j) {
                        *reinterpret_cast<float2 *>(ss + g * SW + 8 * j + 2 * t) = make_float2(d[j][0], d[j][1]);
                        *reinterpret_cast<float2 *>(ss + (g + 8) * SW + 8 * j + 2 * t) = make_float2(d[j][2], d[j][3]);
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        unsigned q = max(top[h], __shfl_xor_sync(0xffffffffu, top[h], 1));
                        q = max(q, __shfl_xor_sync(0xffffffffu, q, 2));
                        if (t == 0) ss[(g + 8 * h) * SW + N] = __uint_as_float(q);
                    }
                }
            }
            const bool act[2] = {tt[0] >= 0 && tt[0] < t_end[0], tt[1] >= 0 && tt[1] < t_end[1]};
            // ---- input half of the gates: u from memory, or x contracted here
            float xr[NT][4], xz[NT][4], xn[NT][4];
            if (proj) {
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int q = 0; q < 4; ++q) { xr[j][q] = 0.0f; xz[j][q] = 0.0f; xn[j][q] = 0.0f; }
                auto ldxs = [&](int k, float2 (&v)[2 * KB]) {    // rows g, g + 8 at columns 2t .. (and 2t + 8 ..)
#pragma unroll
                    for (int q = 0; q < 2 * KB; ++q) v[q] = act[q & 1] ? ldx(xp[q & 1], 8 * KB * k + 8 * (q >> 1) + 2 * t) : make_float2(0.0f, 0.0f);
                };
                float2 xc[2 * KB];
                ldxs(0, xc);
#pragma unroll 1
                for (int kk = 0; kk < kx; ++kk) {
                    unsigned ah[4], al[4];
#pragma unroll
                    for (int q = 0; q < 2 * KB; ++q) operand(ah, al, q >> 1, q & 1, xc[q], *reinterpret_cast<const float2 *>(s_xf + (F16 ? 16 * kk + 8 * (q >> 1) + 2 * t : 0)));
                    if (kk + 1 < kx) ldxs(kk + 1, xc);
                    const uint4 *q0 = sI + (4 * kk + t) * NS + g;
#pragma unroll
                    for (int j = 0; j < NT; ++j) {
#pragma unroll
                        for (int gate = 0; gate < 3; ++gate) {
                            const uint4 w = q0[gate * N + 8 * j];
                            float (&acc)[4] = gate == 0 ? xr[j] : gate == 1 ? xz[j] : xn[j];
                            mma(acc, al, w.x, w.y);
                            mma(acc, ah, w.z, w.w);
                            mma(acc, ah, w.x, w.y);
                        }
                    }
                }
            } else if constexpr (U_AHEAD) {              // (requested a step ago; the next one's now)
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int q = 0; q < 4; ++q) { xr[j][q] = ur_n[j][q]; xz[j][q] = uz_n[j][q]; xn[j][q] = un_n[j][q]; }
                if (step + 1 < s_end) load_u(ur_n, uz_n, un_n, 1);
            } else {
                load_u(xr, xz, xn, 0);
            }
            if (F16 && !proj) {                          // (in the products' scale: a power of two)
                const float up = pow2_inverse(kS);
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int q = 0; q < 4; ++q) { xr[j][q] *= up; xz[j][q] *= up; xn[j][q] *= up; }
            }
            // the state as A operands, and the power of two of p: |p| <= |lambda| / 4 or so, its exponent to 2^9 in every row
            unsigned ah[NB][4], al[NB][4];
            if constexpr (F16 && NT % 2) {
#pragma unroll
                for (int q = 2; q < 4; ++q) { ah[NB - 1][q] = 0u; al[NB - 1][q] = 0u; }
            }
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int h = 0; h < 2; ++h) operand(ah[j / KB], al[j / KB], j % KB, h, make_float2(hp[j][2 * h], hp[j][2 * h + 1]), make_float2(MMA_OP_SCALE, MMA_OP_SCALE));
            float sc[2] = {1.0f, 1.0f}, kM[2] = {1.0f, 1.0f};
            if constexpr (F16) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    unsigned q = 0u;
#pragma unroll
                    for (int j = 0; j < NT; ++j)
                        q = max(q, max(__float_as_uint(fabsf(gy[j][2 * h] + d[j][2 * h])), __float_as_uint(fabsf(gy[j][2 * h + 1] + d[j][2 * h + 1]))));
                    q = max(q, __shfl_xor_sync(0xffffffffu, q, 1));
                    q = max(q, __shfl_xor_sync(0xffffffffu, q, 2));
                    const int ex = min(max((int)(q >> 23), 20), 240);
                    sc[h] = __uint_as_float((unsigned)(127 + 9 - (ex - 127)) << 23);
                    kM[h] = __uint_as_float((unsigned)(127 - 9 + (ex - 127)) << 23) / wscale;
                }
            }
            // ---- hidden half, gates, lambda and the pre-activation gradients, one block of eight columns at a time
            unsigned ph[PB][4], pl[PB][4];               // p as A operands: block gate * NT + j of eight columns
            if constexpr (F16 && 3 * NT % 2) {
#pragma unroll
                for (int q = 2; q < 4; ++q) { ph[PB - 1][q] = 0u; pl[PB - 1][q] = 0u; }
            }
            float zl[NT][4];
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                float (&hr)[4] = xr[j], (&hz)[4] = xz[j];
                float hq[4] = {0.f, 0.f, 0.f, 0.f};
                const uint4 *q0 = sH + t * NS + 8 * j + g;
#pragma unroll
                for (int kk = 0; kk < NB; ++kk)
#pragma unroll
                    for (int gate = 0; gate < 3; ++gate) {
                        const uint4 w = q0[4 * kk * NS + gate * N];
                        float (&acc)[4] = gate == 0 ? hr : gate == 1 ? hz : hq;
                        low(ah[kk], al[kk]);
                        mma(acc, al[kk], w.x, w.y);
                        mma(acc, ah[kk], w.z, w.w);
                        mma(acc, ah[kk], w.x, w.y);
                    }
                const int col = 8 * j + 2 * t;
                const float2 bR = *reinterpret_cast<const float2 *>(sb + col), bZ = *reinterpret_cast<const float2 *>(sb + N + col);
                const float2 bQ = *reinterpret_cast<const float2 *>(sb + 2 * N + col), bN = *reinterpret_cast<const float2 *>(sb + 3 * N + col);
                const float2 one = make_float2(1.0f, 1.0f), mone = make_float2(-1.0f, -1.0f), k2 = make_float2(kS, kS);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float2 h2 = make_float2(hp[j][2 * h], hp[j][2 * h + 1]);
                    const float2 l2 = fadd2(make_float2(gy[j][2 * h], gy[j][2 * h + 1]), make_float2(d[j][2 * h], d[j][2 * h + 1]));
                    const float2 q = ffma2(make_float2(hq[2 * h], hq[2 * h + 1]), k2, bQ);
                    const float2 r = sigmoid2_gate(ffma2(make_float2(hr[2 * h], hr[2 * h + 1]), k2, bR));
                    const float2 z = sigmoid2_gate(ffma2(make_float2(hz[2 * h], hz[2 * h + 1]), k2, bZ));
                    const float2 c = tanh2_gate(ffma2(r, q, ffma2(make_float2(xn[j][2 * h], xn[j][2 * h + 1]), k2, bN)));
                    const float2 omz = ffma2(z, mone, one), omr = ffma2(r, mone, one);
                    const float2 pz = fmul2(fmul2(fmul2(ffma2(c, mone, h2), z), omz), l2);
                    const float2 pa = fmul2(fmul2(omz, ffma2(fmul2(c, mone), c, one)), l2);          // w.r.t. W_in x + b_in
                    const float2 pn = fmul2(pa, r);                                                  // w.r.t. W_hn h + b_hn
                    const float2 pr = fmul2(fmul2(pn, q), omr);
                    const float2 zz = fmul2(z, l2);
                    const float2 pg[3] = {pr, pz, pn};
#pragma unroll
                    for (int gate = 0; gate < 3; ++gate) operand(ph[(gate * NT + j) / KB], pl[(gate * NT + j) / KB], (gate * NT + j) % KB, h, pg[gate], make_float2(sc[h], sc[h]));
                    zl[j][2 * h] = zz.x; zl[j][2 * h + 1] = zz.y;
                    if (step >= burn && act[h]) {
                        if (col < n) mb = max(mb, __float_as_uint(fabsf(l2.x)));
                        if (col + 1 < n) mb = max(mb, __float_as_uint(fabsf(l2.y)));
                        const long long o = row[h] * H + blockIdx.y;
                        auto st2 = [&](float *dst, float2 v) {
                            if constexpr (V2) { if (col < n) *reinterpret_cast<float2 *>(dst) = v; }
                            else { if (col < n) dst[0] = v.x; if (col + 1 < n) dst[1] = v.y; }
                        };
                        if (a.lam) {
                            st2(a.lam + o * n + col, l2);
                        } else if (a.packed) {
                            float *gi = a.dGi + o * 4 * n + col;
                            st2(gi, pr); st2(gi + n, pz); st2(gi + 2 * n, pn); st2(gi + 3 * n, pa);
                        } else {
                            float *gi = a.dGi + o * 3 * n + col, *gh = a.dGh + o * 3 * n + col;
                            st2(gi, pr); st2(gi + n, pz); st2(gi + 2 * n, pa);
                            st2(gh, pr); st2(gh + n, pz); st2(gh + 2 * n, pn);
                        }
                    }
                }
            }
            // ---- advance; the next position's state and dL/dy are requested while p W_h runs
#pragma unroll
            for (int h = 0; h < 2; ++h) { ++tt[h]; row[h] -= s; yp[h] -= ys; gp[h] -= ys; xp[h] -= xs; }
            if (step + 1 < s_end) { load_h(hp); load_g(gy); }
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                float acc[4], cr[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[q] = F16 ? 0.0f : zl[j][q];
                const uint4 *q0 = sT + t * NS2 + 8 * j + g;
#pragma unroll
                for (int kk = 0; kk < PB; ++kk) {
                    const uint4 w = q0[4 * kk * NS2];
                    low(ph[kk], pl[kk]);
                    mma(cr, pl[kk], w.x, w.y);
                    mma(cr, ph[kk], w.z, w.w);
                    mma(acc, ph[kk], w.x, w.y);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) d[j][q] = act[q >> 1] ? (F16 ? fmaf(acc[q] + cr[q], kM[q >> 1], zl[j][q]) : acc[q] + cr[q]) : d[j][q];
            }
        }
        // ---- the state that leaves the first time step: the gradient w.r.t. y0 (wanted or not, it shows what is not finite there)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (t_end[h] > 0 && !next[h]) {
#pragma unroll
                for (int j = 0; j < NT; ++j) mb_end = max(mb_end, max(__float_as_uint(fabsf(d[j][2 * h])), __float_as_uint(fabsf(d[j][2 * h + 1]))));
                if (a.dy0) {
                    const long long q = (grp * 16 + g + 8 * h) / nchain;
                    float *o = a.dy0 + (a.dy0_by_head ? q * H + blockIdx.y : hd.first_seq + q) * n;
#pragma unroll
                    for (int j = 0; j < NT; ++j) {
                        const int col = 8 * j + 2 * t;
                        if (col < n) o[col] = d[j][2 * h];
                        if (col + 1 < n) o[col + 1] = d[j][2 * h + 1];
                    }
                }
            }
        // ---- boundaries: this row's end state against the state its successor assumed
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = g + 8 * h;
            if (next[h] && row < 15) {
                unsigned off = 0u;
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const float2 v = *reinterpret_cast<const float2 *>(ss + (row + 1) * SW + 8 * j + 2 * t);
                    const unsigned q = max(absdiff_bits(v.x, d[j][2 * h]), absdiff_bits(v.y, d[j][2 * h + 1]));
                    off = max(off, q);
                }
                mis = max(mis, off);
                rel = max(rel, boundary_ratio(off, ss[(row + 1) * SW + N]));
                if (near[h]) mis_end = max(mis_end, off);
            }
        }
        const bool near_next = __shfl_sync(0xffffffffu, (int)near[1], 28) != 0;
        const bool has_next = __shfl_sync(0xffffffffu, (int)next[1], 28) != 0;                   // row 15
        const bool has_prev = __shfl_sync(0xffffffffu, (int)(t_end[0] > 0 && grp > 0 && (grp * 16) % nchain != 0), 0) != 0;   // row 0
        __syncwarp();
        if (has_next) {                                  // row 15's end state takes the place of row 15's start state
            if (g == 7) {
#pragma unroll
                for (int j = 0; j < NT; ++j)
                    *reinterpret_cast<float2 *>(ss + 15 * SW + 8 * j + 2 * t) = make_float2(d[j][2], d[j][3]);
            }
        }
        __syncwarp();
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {           // 0: left of the boundary behind this group, 1: right of the one before it
            if (side == 0 ? !has_next : !has_prev) continue;
            const size_t edge = (size_t)hd.first_edge + (size_t)grp - side;
            const float *own = ss + (side == 0 ? 15 : 0) * SW;
            float *slot = a.edge + edge * ADJ_EDGE(n);
            for (int i = lane; i < n; i += 32) __stcg(slot + side * n + i, own[i]);
            if (side == 1 && lane == 0) __stcg(slot + 2 * n, own[N]);
            __threadfence();
            __syncwarp();
            unsigned old = 0;
            if (lane == 0) old = atomicAdd(a.edge_flag + edge, 1u);
            old = __shfl_sync(0xffffffffu, old, 0);
            if (old == 1u) {
                __threadfence();
                const bool near_here = side == 0 ? near_next : near_prev;
                const float scale = side == 0 ? __ldcg(slot + 2 * n) : own[N];
                for (int i = lane; i < n; i += 32) {
                    const unsigned q = absdiff_bits(own[i], __ldcg(slot + (side ^ 1) * n + i));
                    mis = max(mis, q);
                    rel = max(rel, boundary_ratio(q, scale));
                    if (near_here) mis_end = max(mis_end, q);
                }
                if (lane == 0) a.edge_flag[edge] = 0u;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
        mis = max(mis, __shfl_xor_sync(0xffffffffu, mis, o));
        rel = max(rel, __shfl_xor_sync(0xffffffffu, rel, o));
        mb_end = max(mb_end, __shfl_xor_sync(0xffffffffu, mb_end, o));
        mis_end = max(mis_end, __shfl_xor_sync(0xffffffffu, mis_end, o));
    }
    if (lane == 0) {
        if (mb) atomicMax(&st->err_bits, mb);
        if (mis) atomicMax(&st->mis_bits, mis);
        if (rel) atomicMax(&st->rel_bits, rel);
        if (mb_end) atomicMax(&st->top_end_bits, mb_end);
        if (mis_end) atomicMax(&st->mis_end_bits, mis_end);
        __threadfence();
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        const unsigned prev = atomicAdd(&st->exit_counter, 1u);
        if (prev + 1u == nctas) {
            __threadfence();
            st->exit_counter = 0u;
            adjoint_decide(st, a.eta, a.dy0 != nullptr, burn);
        }
    }
}

}  // namespace deer
