// One Newton body of deer_gru_eval (Eq. 3 with Eq. 5, Newton-update form of App. A.1) as ONE launch: cell, residual,
// linear solve, new iterate and convergence maximum, with nothing but x, the old iterate and the new one in memory.
//
// The update solves d_t = J_t d_{t-1} + r_t, r_t = f(y_{t-1}, x_t) - y_t.  The sequences are cut into chains of L
// positions; sixteen chains advance in lockstep as the sixteen rows of a warp's m16n8k16 MMAs, a step being
//     [16, m] x [m, 3n] + [16, n] x [n, 3n]      gates: hi + lo f16 halves in three MMAs, so f is good to fp32 level
//     [16, n] x [n, 3n]                          J_t d_{t-1} = z.d + k_r.(W_hr d) + a_z.(W_hz d) + k_n.(W_hn d)
// with the gate arithmetic elementwise on the accumulator fragments.  The accumulator fragments of two blocks of eight
// columns are the A operand of a K step of 16 as they stand, so neither J_t, nor its coefficients, nor any chain product
// is ever formed or stored.  Powers of two (operand_scales, MMA_D_SCALE) keep the halves among the normal f16 numbers; a
// value beyond f16's range makes a NaN, and the body is run again with projected inputs, or is for the other kernels.
//
// What a chain does not know is the update entering it.  It starts `burn` positions early from zero: the error of its
// entering update is the old error carried through `burn` Jacobians, and the Jacobians of a cell that forgets make it
// vanish.  That is not taken on trust: every chain's end state is compared with the state its successor had assumed at
// the same position (same arithmetic on same inputs: the difference is the carried error and nothing else).  The
// largest mismatch of the launch has to stay below eta * max(err, tol) -- the accuracy the linear solve is asked for
// in any case, since the fixed point does not depend on it.  When it does not, the body is not counted: the burn-in is
// raised to what the observed decay calls for and the body is run again, or, for a cell that hardly forgets, the
// evaluation goes on with the kernels that multiply the Jacobians out (BODY_FALL_BACK).
//
// What bounds it: the latency of a step's MMAs and gates with eight warps per SM.  n = 28, m = 8, B = 16, T = 2e4: tensor pipe 35 %
// active, issue slots 32 % used, DRAM 3 %.
//
// Nothing waits on another CTA.  Boundaries inside a warp are compared from shared memory; at a boundary between two
// warps each side leaves its state in global memory and the one that arrives second compares.
#pragma once
#include "mma_tf32.cuh"
#include "newton_body.h"
#include "split_f16.cuh"

namespace deer {

// End of a body that is a launch of its own: the last CTA's decision.  unit: what the launch rounds its burn-in up to
// (a rate that is not adapted to may be underestimated); narrow: its products hold what f16 does.  Single thread.
__device__ __forceinline__ void body_decide(StatusBlock *st, const BodyArgs &a, int unit = 1, float rounding = 0.0f, bool narrow = false)
{
    const float e = __uint_as_float(*(volatile unsigned *)&st->err_bits);
    const float mis = __uint_as_float(*(volatile unsigned *)&st->mis_bits);
    if (narrow && (!(e <= 3.402823466e38f) || !(mis <= 3.402823466e38f))) {
        st->err_bits = 0u; st->mis_bits = 0u;
        st->burn = 0;
        st->done = BODY_BEYOND;
        if (HostResult *h = st->host) { h->burn = 0; post_done(h, BODY_BEYOND); }
        return;
    }
    const BodyVerdict v = body_verdict(e, mis, a.eta, a.adapt ? (st->burn + unit - 1) / unit * unit : st->burn, a.burn_cap, a.T, st->tol, st->iters, st->max_iter, a.adapt != 0, rounding);
    st->mis_bits = 0u;
    if (v.need) st->need = max(st->need, v.need);
    st->burn = v.done == BODY_DONE ? st->need : v.burn;
    if (v.counts) newton_decide(st, st->tol, st->max_iter, st->trace, a.polled != 0);
    if (v.counts && (st->done || !v.done)) return;
    st->err_bits = 0u;
    st->done = v.done;
    if (HostResult *h = st->host) { h->burn = v.burn; if (v.done) post_done(h, v.done); }
}

// Scales of the states (values up to 16,376; what is below 2^-5 of one keeps 2^-27 absolute: they come from gates that are good to
// 2e-7) and of the update (up to 1,023, as behind a y0 of some hundred; 2^-31 absolute: the last body's is the tolerance or less) as
// f16 operands, and of a channel's largest weight (operand_scales).
constexpr float MMA_OP_SCALE = 4.0f, MMA_D_SCALE = 64.0f;
constexpr int MMA_TOP = 10;

template <int N> struct Body {
    static constexpr int NT = N / 8, NB = (NT + 1) / 2;  // column blocks, K steps
    static constexpr int NS = 3 * N + 2;                 // records per lane of a K step: = 2 (mod 8), conflict-free
    static constexpr int SW = N + 4;                     // stride of a saved start state
    static constexpr size_t smem(int warps, int kx)      // kx: 8-column blocks of x contracted in the kernel
    {
        return sizeof(float) * ((size_t)16 * (NB + (kx + 1) / 2) * NS + 4 * N + (size_t)warps * 16 * SW);
    }
};

// EXACT: the products with d are three MMAs as well (sizes whose solve has always been fp32-accurate); V2: rows are read and
// written as 8-byte pairs.  n <= 8 takes a thread per chain instead (newton_lane.cuh).
// (Two CTAs per SM from n = 17 to 32, not three: 168 registers spill.  us per evaluation, three / two: n = 20, 480,000 positions 739 /
// 649; n = 28, 320,000 832 / 635; n = 30, m = 30, 480,000 1181 / 1033.)
template <int N, bool V2, bool EXACT>
__global__ void __launch_bounds__(N > 32 ? 256 : 128, N > 32 ? 1 : N > 16 ? 2 : 3) newton_body_kernel(BodyArgs a)
{
    using C = Body<N>;
    constexpr int NT = C::NT, NB = C::NB, NS = C::NS, SW = C::SW;
    extern __shared__ __align__(16) float smb[];
    __shared__ unsigned s_top;
    __shared__ __align__(16) float s_xf[64];
    const BodyHead hd = a.heads ? a.heads[blockIdx.y] : a.h0;
    StatusBlock *st = a.st + blockIdx.y;
    const int n = a.n, m = a.m, H = a.H, L = a.L;
    const bool proj = a.u == nullptr;
    const int kx = proj ? (m + 15) >> 4 : 0;             // K steps of x
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int g = lane >> 2, t = lane & 3;

    // geometry of this CTA's head
    const int s = hd.stride, Tp = (a.T + s - 1) / s, nchain = (Tp + L - 1) / L;
    const long long total = (long long)a.B * s * nchain;
    const long long groups = (total + 15) >> 4;
    const unsigned nctas = (unsigned)((groups + nwarps - 1) / nwarps);
    if (blockIdx.x >= nctas) return;

    // ---- weights into shared memory as records of the four words that a lane needs for a column of a K step: hi of rows 2t, 2t + 1
    // and 2t + 8, 2t + 9, and lo of the same: one 128-bit load (weights are not produced by the previous launch: this runs before
    // its end)
    uint4 *sH = reinterpret_cast<uint4 *>(smb), *sI = sH + 4 * NB * NS;
    float *sb = reinterpret_cast<float *>(sI + 4 * kx * NS);
    const float wscale = operand_scales(hd.W_h, hd.W_i, 3 * n, n, proj ? m : 0, MMA_OP_SCALE, MMA_TOP, s_xf, &s_top);
    const float unit = wscale * MMA_OP_SCALE, kS = 1.0f / unit, kD = 1.0f / (wscale * MMA_D_SCALE);
    auto record = [&](const float *wr, bool row, int kt, int width, auto scale) {
        const int k = 16 * (kt >> 2) + 2 * (kt & 3);
        auto w = [&](int j) { return row && j < width ? wr[j] * scale(j) : 0.0f; };
        uint4 r;
        split_f16(make_float2(w(k), w(k + 1)), r.x, r.z);
        split_f16(make_float2(w(k + 8), w(k + 9)), r.y, r.w);
        return r;
    };
    for (int idx = tid; idx < 4 * NB * 3 * N; idx += blockDim.x) {
        const int kt = idx % (4 * NB), c = idx / (4 * NB), gate = c / N, i = c % N;
        sH[kt * NS + c] = record(hd.W_h + (size_t)(gate * n + i) * n, i < n, kt, n, [&](int) { return wscale; });
    }
    for (int idx = tid; idx < 4 * kx * 3 * N; idx += blockDim.x) {
        const int kt = idx % (4 * kx), c = idx / (4 * kx), gate = c / N, i = c % N;
        sI[kt * NS + c] = record(hd.W_i + (size_t)(gate * n + i) * m, i < n, kt, m, [&](int j) { return unit * pow2_inverse(s_xf[j]); });
    }
    for (int i = tid; i < N; i += blockDim.x) {          // (u holds b_i already)
        sb[i] = i < n ? hd.b_h[i] + (proj ? hd.b_i[i] : 0.0f) : 0.0f;
        sb[N + i] = i < n ? hd.b_h[n + i] + (proj ? hd.b_i[n + i] : 0.0f) : 0.0f;
        sb[2 * N + i] = i < n ? hd.b_h[2 * n + i] : 0.0f;
        sb[3 * N + i] = i < n && proj ? hd.b_i[2 * n + i] : 0.0f;
    }
    float *ss = sb + 4 * N + warp * 16 * SW;             // start states of this warp's chains
    pdl_prologue();
    if (*(volatile int *)&st->done) return;
    __syncthreads();

    const int iters = *(volatile int *)&st->iters, burn = *(volatile int *)&st->burn;
    const float *ycur = a.buf[iters & 1];
    const ptrdiff_t to_new = a.buf[(iters + 1) & 1] - ycur;
    const bool zero = iters == 0 && !a.warm;             // the guess is zero: nothing of it is read
    const long long grp = (long long)blockIdx.x * nwarps + warp;
    unsigned mb = 0u, mis = 0u;

    if (grp < groups) {
        // ---- rows g and g + 8 of this lane: chain c of sequence (b, phase)
        int tt[2], t_end[2];
        const float *yp[2], *xp[2], *y0p[2];             // pointers at position tt (not dereferenced outside the sequence)
        bool next[2];                                    // the row's chain has a successor
        const size_t ys = (size_t)s * H * n, xs = proj ? (size_t)s * m : (size_t)s * H * 3 * n;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const long long gid = grp * 16 + g + 8 * h;
            const long long q = gid < total ? gid / nchain : 0;
            const int c = gid < total ? (int)(gid - q * nchain) : 0;
            const long long b = q / s;
            const int ph = (int)(q - b * s);
            const int len = gid < total ? (a.T - ph + s - 1) / s : 0;
            t_end[h] = min(len, (c + 1) * L);
            if (c * L >= len) t_end[h] = 0;
            next[h] = (c + 1) * L < len;
            tt[h] = c * L - burn;
            const size_t e = (size_t)b * a.T + ph;
            yp[h] = ycur + (e * H + blockIdx.y) * n + (ptrdiff_t)tt[h] * (ptrdiff_t)ys;
            xp[h] = (proj ? a.x + e * m : a.u + (e * H + blockIdx.y) * 3 * n) + (ptrdiff_t)tt[h] * (ptrdiff_t)xs;
            y0p[h] = a.y0 + ((size_t)b * H + blockIdx.y) * n;
        }
        // (a warp whose chains are all first ones has no burn-in: its earliest position is -burn)
        const int tmax = __reduce_max_sync(0xffffffffu, max(t_end[0] > 0 ? tt[0] : -burn, t_end[1] > 0 ? tt[1] : -burn));
        const int s_first = tmax <= -burn ? burn : 0;
        const int s_end = __reduce_max_sync(0xffffffffu, max(t_end[0] > 0 ? t_end[0] - tt[0] : 0, t_end[1] > 0 ? t_end[1] - tt[1] : 0));
#pragma unroll
        for (int h = 0; h < 2; ++h) { tt[h] += s_first; yp[h] += (ptrdiff_t)s_first * (ptrdiff_t)ys; xp[h] += (ptrdiff_t)s_first * (ptrdiff_t)xs; }

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
        // iterate at position tt + off of row h (off = -1, 0): y0 before the first position, zero where nothing is
        auto load_y = [&](float (&dst)[NT][4], int off) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int q = tt[h] + off;
                const bool in = q >= 0 && q < t_end[h] && !zero, first = q == -1 && t_end[h] > 0;
                const float *p = first ? y0p[h] : yp[h] + (ptrdiff_t)off * (ptrdiff_t)ys;
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const float2 v = in || first ? ld2(p, 8 * j + 2 * t, n) : make_float2(0.0f, 0.0f);
                    dst[j][2 * h] = v.x; dst[j][2 * h + 1] = v.y;
                }
            }
        };
        float hp[NT][4], yc[NT][4], d[NT][4];
        load_y(hp, -1);
        load_y(yc, 0);
#pragma unroll
        for (int j = 0; j < NT; ++j) { d[j][0] = d[j][1] = d[j][2] = d[j][3] = 0.0f; }

        // projected inputs at position tt + ahead
        constexpr bool U_AHEAD = NT <= 2;                // a step ahead where the registers allow it
        auto load_u = [&](float (&vr)[NT][4], float (&vz)[NT][4], float (&vn)[NT][4], int ahead) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool on = tt[h] + ahead >= 0 && tt[h] + ahead < t_end[h];
                const float *q = xp[h] + ahead * (ptrdiff_t)xs;
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

#pragma unroll 1
        for (int step = s_first; step < s_end; ++step) {
            if (step == burn) {
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    *reinterpret_cast<float2 *>(ss + g * SW + 8 * j + 2 * t) = make_float2(d[j][0], d[j][1]);
                    *reinterpret_cast<float2 *>(ss + (g + 8) * SW + 8 * j + 2 * t) = make_float2(d[j][2], d[j][3]);
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
                auto ldxs = [&](int k, float2 (&v)[4]) {         // rows g, g + 8 at columns 2t .. and 2t + 8 ..
#pragma unroll
                    for (int q = 0; q < 4; ++q) v[q] = act[q & 1] ? ldx(xp[q & 1], 16 * k + 8 * (q >> 1) + 2 * t) : make_float2(0.0f, 0.0f);
                };
                float2 xc[4];
                ldxs(0, xc);
#pragma unroll 1
                for (int kk = 0; kk < kx; ++kk) {
                    unsigned ah[4], al[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) split_f16(fmul2(xc[q], *reinterpret_cast<const float2 *>(s_xf + 16 * kk + 8 * (q >> 1) + 2 * t)), ah[q], al[q]);
                    if (kk + 1 < kx) ldxs(kk + 1, xc);
                    const uint4 *q0 = sI + (4 * kk + t) * NS + g;
#pragma unroll
                    for (int j = 0; j < NT; ++j)
#pragma unroll
                        for (int gate = 0; gate < 3; ++gate) {
                            const uint4 w = q0[gate * N + 8 * j];
                            float (&acc)[4] = gate == 0 ? xr[j] : gate == 1 ? xz[j] : xn[j];
                            mma_f16(acc, al, w.x, w.y);
                            mma_f16(acc, ah, w.z, w.w);
                            mma_f16(acc, ah, w.x, w.y);
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
            if (!proj) {                                 // (in the products' scale: a power of two)
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int q = 0; q < 4; ++q) { xr[j][q] *= unit; xz[j][q] *= unit; xn[j][q] *= unit; }
            }
            // ---- hidden half and the update, one block of eight columns at a time
            const bool hid = !zero || __any_sync(0xffffffffu, tt[0] == 0 || tt[1] == 0);     // zero guess: W_h 0 = 0
            unsigned ah[NB][4], al[NB][4], dh[NB][4], dl[NB][4];
#pragma unroll
            for (int k = 0; k < NB; ++k)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int j = 2 * k + (q >> 1), e = 2 * (q & 1);
                    if (j < NT) {
                        const int jj = j < NT ? j : 0;
                        split_f16(fmul2(make_float2(hp[jj][e], hp[jj][e + 1]), make_float2(MMA_OP_SCALE, MMA_OP_SCALE)), ah[k][q], al[k][q]);
                        const float2 ds = fmul2(make_float2(d[jj][e], d[jj][e + 1]), make_float2(MMA_D_SCALE, MMA_D_SCALE));
                        if constexpr (EXACT) split_f16(ds, dh[k][q], dl[k][q]);
                        else { dh[k][q] = pack_f16(ds); dl[k][q] = 0u; }
                    } else {
                        ah[k][q] = 0u; al[k][q] = 0u; dh[k][q] = 0u; dl[k][q] = 0u;
                    }
                }
            float dn[NT][4];
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                {
                    float hr[4] = {xr[j][0], xr[j][1], xr[j][2], xr[j][3]}, hz[4] = {xz[j][0], xz[j][1], xz[j][2], xz[j][3]};
                    float hq[4] = {0.f, 0.f, 0.f, 0.f}, ur[4] = {0.f, 0.f, 0.f, 0.f}, uz[4] = {0.f, 0.f, 0.f, 0.f}, un[4] = {0.f, 0.f, 0.f, 0.f};
                    const uint4 *q0 = sH + t * NS + 8 * j + g;
#pragma unroll
                    for (int kk = 0; kk < NB; ++kk)
#pragma unroll
                        for (int gate = 0; gate < 3; ++gate) {
                            const uint4 w = q0[4 * kk * NS + gate * N];
                            float (&hacc)[4] = gate == 0 ? hr : gate == 1 ? hz : hq;
                            float (&uacc)[4] = gate == 0 ? ur : gate == 1 ? uz : un;
                            if (hid) {
                                mma_f16(hacc, al[kk], w.x, w.y);
                                mma_f16(hacc, ah[kk], w.z, w.w);
                                mma_f16(hacc, ah[kk], w.x, w.y);
                            }
                            if constexpr (EXACT) {
                                mma_f16(uacc, dl[kk], w.x, w.y);
                                mma_f16(uacc, dh[kk], w.z, w.w);
                            }
                            mma_f16(uacc, dh[kk], w.x, w.y);
                        }
                    const int col = 8 * j + 2 * t;
                    const float2 bR = *reinterpret_cast<const float2 *>(sb + col), bZ = *reinterpret_cast<const float2 *>(sb + N + col);
                    const float2 bQ = *reinterpret_cast<const float2 *>(sb + 2 * N + col), bN = *reinterpret_cast<const float2 *>(sb + 3 * N + col);
                    const float2 one = make_float2(1.0f, 1.0f), mone = make_float2(-1.0f, -1.0f), k2 = make_float2(kS, kS);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float2 h2 = make_float2(hp[j][2 * h], hp[j][2 * h + 1]), y2 = make_float2(yc[j][2 * h], yc[j][2 * h + 1]);
                        const float2 d2 = make_float2(d[j][2 * h], d[j][2 * h + 1]);
                        const float2 q = ffma2(make_float2(hq[2 * h], hq[2 * h + 1]), k2, bQ);
                        const float2 r = sigmoid2_gate(ffma2(make_float2(hr[2 * h], hr[2 * h + 1]), k2, bR));
                        const float2 z = sigmoid2_gate(ffma2(make_float2(hz[2 * h], hz[2 * h + 1]), k2, bZ));
                        const float2 c = tanh2_gate(ffma2(r, q, ffma2(make_float2(xn[j][2 * h], xn[j][2 * h + 1]), k2, bN)));
                        const float2 omz = ffma2(z, mone, one), omr = ffma2(r, mone, one);
                        const float2 f = ffma2(omz, c, fmul2(z, h2));
                        const float2 az = fmul2(fmul2(ffma2(c, mone, h2), z), omz);
                        const float2 an = fmul2(omz, ffma2(fmul2(c, mone), c, one));
                        const float2 kn = fmul2(an, r);
                        const float2 kr = fmul2(fmul2(kn, q), omr);
                        float2 v = ffma2(y2, mone, f);                                          // r_t = f - y
                        v = ffma2(z, d2, v);
                        float2 s = fmul2(kr, make_float2(ur[2 * h], ur[2 * h + 1]));
                        s = ffma2(az, make_float2(uz[2 * h], uz[2 * h + 1]), s);
                        s = ffma2(kn, make_float2(un[2 * h], un[2 * h + 1]), s);
                        v = ffma2(s, make_float2(kD, kD), v);
                        dn[j][2 * h] = v.x; dn[j][2 * h + 1] = v.y;
                        if (step >= burn && act[h]) {
                            const float2 yn = fadd2(y2, v);
                            float *o = const_cast<float *>(yp[h]) + to_new + col;
                            if constexpr (V2) {
                                if (col < n) {
                                    mb = max(mb, max(absdiff_bits(yn.x, y2.x), absdiff_bits(yn.y, y2.y)));
                                    *reinterpret_cast<float2 *>(o) = yn;
                                }
                            } else {
                                if (col < n) { mb = max(mb, absdiff_bits(yn.x, y2.x)); o[0] = yn.x; }
                                if (col + 1 < n) { mb = max(mb, absdiff_bits(yn.y, y2.y)); o[1] = yn.y; }
                            }
                        }
                    }
                }
            }
            // ---- advance
#pragma unroll
            for (int h = 0; h < 2; ++h) { ++tt[h]; yp[h] += ys; xp[h] += xs; }
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        d[j][q] = act[q >> 1] ? dn[j][q] : d[j][q];
                        hp[j][q] = yc[j][q];
                    }
                }
            }
            if (step + 1 < s_end) load_y(yc, 0);
        }
        // ---- boundaries: this row's end state against the state its successor assumed
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = g + 8 * h;
            if (next[h] && row < 15) {
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const float2 v = *reinterpret_cast<const float2 *>(ss + (row + 1) * SW + 8 * j + 2 * t);
                    mis = max(mis, max(absdiff_bits(v.x, d[j][2 * h]), absdiff_bits(v.y, d[j][2 * h + 1])));
                }
            }
        }
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
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
        mis = max(mis, __shfl_xor_sync(0xffffffffu, mis, o));
    }
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
            body_decide(st, a, 1, 0.0f, true);
        }
    }
}

}  // namespace deer
