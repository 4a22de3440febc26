// One Newton body as one launch for small states (n up to 8): the solve of newton_body.cuh (chains with a burn-in, boundaries
// verified; see there) with ONE THREAD per chain, everything in fp32 registers.
//
// An 8-column MMA tile is mostly padding at n = 1, 2, 4, and even at n = 8 the split products cost more issue slots than
// plain FMAs with the weights as broadcast 16-byte loads.  A warp's 32 chains walk in lockstep through windows of W positions
// that cp.async has brought into warp-private shared memory (full lines of every chain, one window ahead); the new iterate
// replaces the old one there and leaves the same way.  Row strides are odd in 16-byte pieces: conflict-free.
// What bounds it: issue slots and latency.  n = m = 1, B = 16, T = 3e5, at 94 registers (20 warps fit an SM, 14 were active on average;
// now 108, 16 fit): issue slots 54 % used, special functions (six instructions per state component) 32 %, FMA 31 %, DRAM 12 %.
#pragma once
#include "newton_body.cuh"
#include "scan_onepass.cuh"

namespace deer {

template <int N, int M> struct Lane {                    // M: input channels, padded (1, 2, 4, 8), or 0: projected inputs u
    static constexpr int WARPS = 4, THREADS = 128;
    static constexpr int XW = M > 0 ? M : 3 * N;         // floats of input per position
    static constexpr int W0 = M > 0 ? (N <= 2 ? 16 : 32) / (N > M ? N : M) : 16 / N;
    static constexpr int W = N == 1 && W0 < 4 ? 4 : W0;  // positions of a window
    static constexpr int P = N < 4 ? 4 / N : 1;          // positions per 16 bytes of state
    static constexpr int Q = N == 1 && W % 8 == 0 ? 8 : N == 1 ? 4 : N == 2 ? (W % 4 == 0 ? 4 : 2) : N == 4 ? 2 : 1;      // positions whose cells are evaluated side by side
    __host__ __device__ static constexpr int stride(int w) { return (((w + 3) / 4) | 1) * 4; }
    static constexpr int YR = stride(W * N), XR = stride(W * XW);
    static constexpr int ROW = 3 * N + 3 * M + 4;        // weights and biases of a state component, padded to 16 bytes
    static constexpr int ROWP = (ROW + 3) / 4 * 4;
    static constexpr size_t SMEM = sizeof(float) * ((size_t)N * ROWP + (size_t)WARPS * 2 * 32 * (YR + XR));
    static_assert(W % P == 0 && W % Q == 0 && Q * N % 4 == 0, "windows are whole pieces");
};

// (A CTA per SM named: the compiler, which left to itself aims at more of them, then keeps the cells of the positions that are
// evaluated side by side in registers.  us per evaluation, without and with: n = m = 1 (1.6e7 positions, four draws) 413 -> 362,
// 305 -> 299, 292 -> 286 and 306 -> 301, the last no more than two runs of one side differ; n = 1, m = 5 616 -> 574, n = 2, m = 4
// 272 -> 252; n = 2, m = 8 229 -> 231 and n = 1 with projected inputs 448 -> 451, which stay without, as do n = 4 and 8: no difference.
// Three CTAs named cost n = 4 and 8 spills, 606 -> 837 us.)
template <int N, int M>
__global__ void __launch_bounds__(128, N <= 2 && M > 0 && N * M <= 8 ? 1 : 0) newton_lane_kernel(BodyArgs a)
{
    using C = Lane<N, M>;
    constexpr int W = C::W, P = C::P, YR = C::YR, XR = C::XR, XW = C::XW, ROWP = C::ROWP, Q = C::Q;
    constexpr float LOG2E = 1.4426950408889634f;
    extern __shared__ __align__(16) float smb[];
    const BodyHead hd = a.heads ? a.heads[blockIdx.y] : a.h0;
    StatusBlock *st = a.st + blockIdx.y;
    const int n = a.n, m = a.m, H = a.H, L = a.L, T = a.T;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int s = hd.stride, Tp = (T + s - 1) / s, nchain = (Tp + L - 1) / L;
    const long long total = (long long)a.B * s * nchain;
    const unsigned nctas = (unsigned)((total + C::THREADS - 1) / C::THREADS);
    if (blockIdx.x >= nctas) return;

    // ---- weights: row i = {W_hr[i], W_hz[i], W_hn[i], W_ir[i], W_iz[i], W_in[i], b_r, b_z, b_hn, b_in}
    float *sw = smb;
    for (int idx = tid; idx < N * ROWP; idx += C::THREADS) {
        const int i = idx / ROWP, k = idx % ROWP;
        float v = 0.0f;
        if (i < n) {
            if (k < 3 * N) { const int g = k / N, c = k % N; if (c < n) v = hd.W_h[(g * n + i) * n + c]; }
            else if (k < 3 * N + 3 * M) { const int g = (k - 3 * N) / (M > 0 ? M : 1), c = (k - 3 * N) % (M > 0 ? M : 1); if (c < m) v = hd.W_i[(size_t)(g * n + i) * m + c]; }
            else if (k == 3 * N + 3 * M) v = hd.b_h[i] + (M > 0 ? hd.b_i[i] : 0.0f);
            else if (k == 3 * N + 3 * M + 1) v = hd.b_h[n + i] + (M > 0 ? hd.b_i[n + i] : 0.0f);
            else if (k == 3 * N + 3 * M + 2) v = hd.b_h[2 * n + i];
            else if (k == 3 * N + 3 * M + 3) v = M > 0 ? hd.b_i[2 * n + i] : 0.0f;
        }
        sw[idx] = v;
    }
    float *ring = smb + N * ROWP + warp * 2 * 32 * (YR + XR);            // two stages: states, inputs
    for (int i = lane; i < 2 * 32 * (YR + XR); i += 32) ring[i] = 0.0f;   // (columns past n and m stay zero)
    pdl_prologue();
    if (*(volatile int *)&st->done) return;
    __syncthreads();

    const int iters = *(volatile int *)&st->iters;
    const int burn = (*(volatile int *)&st->burn + W - 1) / W * W;       // (whole windows)
    const float *ycur = a.buf[iters & 1];
    float *ynew = a.buf[(iters + 1) & 1];
    const bool zero = iters == 0 && !a.warm;             // the guess is zero: nothing of it is read

    // ---- this lane's chain
    const long long gid = ((long long)blockIdx.x * C::WARPS + warp) * 32 + lane;
    const long long q = gid < total ? gid / nchain : 0;
    const int c = gid < total ? (int)(gid - q * nchain) : 0;
    const long long b = q / s;
    const int ph = (int)(q - b * s);
    const int len = gid < total ? (T - ph + s - 1) / s : 0;
    const int te = c * L < len ? min(len, (c + 1) * L) : 0, ts = c * L - burn;
    const bool next = te > 0 && (c + 1) * L < len;
    const long long e0 = b * T + ph + (long long)ts * s; // row in [B,T] of window position 0
    const long long rows = (long long)a.B * T;
    const long long yps = (long long)s * H * n, ups = (long long)s * (M > 0 ? m : H * 3 * n);        // floats between positions
    const float *in = M > 0 ? a.x : a.u;
    // 16-byte copies where every chain's pieces are aligned and dense
    const bool y16 = n == N && (N >= 4 ? true : yps == N && (T * N) % 4 == 0) && (((uintptr_t)ycur | (uintptr_t)ynew) & 15) == 0;
    const bool x16 = M > 0 ? m == M && (M >= 4 ? true : s == 1 && (T * M) % 4 == 0) && ((uintptr_t)in & 15) == 0
                           : n == N && (N >= 4 ? true : ups == 3 * N && (T * 3 * N) % 4 == 0 && W * 3 * N % 4 == 0) && ((uintptr_t)in & 15) == 0;
    const bool idle = __all_sync(0xffffffffu, te == 0);

    // copies of window w (positions W w ..) of all 32 chains; 16 bytes or 4 at a time, consecutive lanes along a chain
    auto fetch = [&](int w) {
        float *sy = ring + (w & 1) * 32 * (YR + XR), *sx = sy + 32 * YR;
        const bool wy = !zero;
        if (wy && y16) {
            constexpr int PC = W * N / 4;                // pieces of a row
#pragma unroll
            for (int i = 0; i < PC; ++i) {
                const int r = (i * 32 + lane) / PC, pc = (i * 32 + lane) % PC;
                const long long er = __shfl_sync(0xffffffffu, e0, r);
                const int pos = W * w + pc * 4 / N;
                const long long e = er + (long long)pos * s;
                if (e >= 0 && e + (P - 1) < rows) cp_async16(sy + r * YR + 4 * pc, ycur + (e * H + blockIdx.y) * n + pc * 4 % N);
            }
        } else if (wy) {
            for (int i = lane; i < 32 * W * N; i += 32) {
                const int r = i / (W * N), f = i % (W * N), col = f % N;
                const long long er = __shfl_sync(0xffffffffu, e0, r);
                const long long e = er + (long long)(W * w + f / N) * s;
                if (e >= 0 && e < rows && col < n) cp_async4(sy + r * YR + f, ycur + (e * H + blockIdx.y) * n + col);
            }
        }
        if (x16) {
            constexpr int PC = W * XW / 4;
#pragma unroll
            for (int i = 0; i < PC; ++i) {
                const int r = (i * 32 + lane) / PC, pc = (i * 32 + lane) % PC;
                const long long er = __shfl_sync(0xffffffffu, e0, r);
                const long long e = er + (long long)(W * w + pc * 4 / XW) * s;
                if (e >= 0 && e + (XW < 4 ? 4 / XW - 1 : 0) < rows) cp_async16(sx + r * XR + 4 * pc, in + (M > 0 ? e * m : (e * H + blockIdx.y) * 3 * n) + pc * 4 % XW);
            }
        } else {
            for (int i = lane; i < 32 * W * XW; i += 32) {
                const int r = i / (W * XW), f = i % (W * XW), col = f % XW;
                const long long er = __shfl_sync(0xffffffffu, e0, r);
                const long long e = er + (long long)(W * w + f / XW) * s;
                const bool ok = M > 0 ? col < m : col % N < n;
                if (e >= 0 && e < rows && ok)
                    cp_async4(sx + r * XR + f, in + (M > 0 ? e * m + col : (e * H + blockIdx.y) * 3 * n + (col / N) * n + col % N));
            }
        }
        cp_async_commit();
    };
    // rows of window w, from the first own position on, to the new iterate
    auto put = [&](int w) {
        const float *sy = ring + (w & 1) * 32 * (YR + XR);
        if (y16) {
            constexpr int PC = W * N / 4;
#pragma unroll
            for (int i = 0; i < PC; ++i) {
                const int r = (i * 32 + lane) / PC, pc = (i * 32 + lane) % PC;
                const long long er = __shfl_sync(0xffffffffu, e0, r);
                const int pos = W * w + pc * 4 / N, t = __shfl_sync(0xffffffffu, ts, r) + pos, end = __shfl_sync(0xffffffffu, te, r);
                float *dst = ynew + ((er + (long long)pos * s) * H + blockIdx.y) * n + pc * 4 % N;
                const float4 v = *reinterpret_cast<const float4 *>(sy + r * YR + 4 * pc);
                if (t + P <= end) *reinterpret_cast<float4 *>(dst) = v;
                else if constexpr (P > 1) {
                    const float e4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) if (t + k / N < end) dst[k] = e4[k];
                }
            }
        } else {
            for (int i = lane; i < 32 * W * N; i += 32) {
                const int r = i / (W * N), f = i % (W * N), col = f % N;
                const long long er = __shfl_sync(0xffffffffu, e0, r);
                const int pos = W * w + f / N, t = __shfl_sync(0xffffffffu, ts, r) + pos, end = __shfl_sync(0xffffffffu, te, r);
                if (t < end && col < n) ynew[((er + (long long)pos * s) * H + blockIdx.y) * n + col] = sy[r * YR + f];
            }
        }
    };

    float h[N], d[N], start[N];
#pragma unroll
    for (int k = 0; k < N; ++k) { h[k] = 0.0f; d[k] = 0.0f; start[k] = 0.0f; }
    if (te > 0) {                                        // the state before the first position
        const float *p = ts >= 1 ? (zero ? nullptr : ycur + ((e0 - s) * H + blockIdx.y) * n) : a.y0 + (b * H + blockIdx.y) * n;
        if (p) {
#pragma unroll
            for (int k = 0; k < N; ++k) if (k < n) h[k] = p[k];
        }
    }
    // weights of small cells in registers, of larger ones from shared memory (broadcast)
    constexpr bool REG = N * ROWP <= 72;
    float4 wreg[REG ? N * ROWP / 4 : 1];
    if constexpr (REG) {
#pragma unroll
        for (int k = 0; k < N * ROWP / 4; ++k) wreg[k] = reinterpret_cast<const float4 *>(sw)[k];
    }

    unsigned mb = 0u;
    const int w0 = nchain == 1 ? burn / W : 0;           // (every chain is a first one: no burn-in)
    const int w_end = idle ? w0 : (burn + min(L, (Tp + W - 1) / W * W)) / W;
    if (w0 < w_end) fetch(w0);
#pragma unroll 1
    for (int w = w0; w < w_end; ++w) {
        if (w + 1 < w_end) fetch(w + 1); else cp_async_commit();
        cp_async_wait_1();
        __syncwarp();
        if (W * w == burn) {
#pragma unroll
            for (int k = 0; k < N; ++k) start[k] = d[k];
        }
        float *sy = ring + (w & 1) * 32 * (YR + XR) + lane * YR;
        const float *sx = ring + (w & 1) * 32 * (YR + XR) + 32 * YR + lane * XR;
#pragma unroll 1
        for (int i0 = 0; i0 < W; i0 += Q) {
            float yv[Q * N], xv[Q * XW];
#pragma unroll
            for (int k = 0; k < Q * N / 4; ++k) {
                const float4 v = zero ? make_float4(0.f, 0.f, 0.f, 0.f) : *reinterpret_cast<const float4 *>(sy + i0 * N + 4 * k);
                yv[4 * k] = v.x; yv[4 * k + 1] = v.y; yv[4 * k + 2] = v.z; yv[4 * k + 3] = v.w;
            }
            if constexpr (Q * XW % 4 == 0) {
#pragma unroll
                for (int k = 0; k < Q * XW / 4; ++k) {
                    const float4 v = *reinterpret_cast<const float4 *>(sx + i0 * XW + 4 * k);
                    xv[4 * k] = v.x; xv[4 * k + 1] = v.y; xv[4 * k + 2] = v.z; xv[4 * k + 3] = v.w;
                }
            } else {
#pragma unroll
                for (int k = 0; k < Q * XW; ++k) xv[k] = sx[i0 * XW + k];
            }
            const int t0 = ts + W * w + i0;
            const bool own = W * w >= burn;
            // The cells of the Q positions depend on the old iterate only: side by side.  z, k_r, k_z, k_n, f of position p,
            // component i; one component at a time, its weights from registers or shared memory (broadcast).
            float cz[Q][N], ckr[Q][N], ckz[Q][N], ckn[Q][N], cf[Q][N];
            float hq[Q][N];
#pragma unroll
            for (int p = 0; p < Q; ++p)
#pragma unroll
                for (int k = 0; k < N; ++k) hq[p][k] = p == 0 ? h[k] : t0 + p - 1 >= 0 ? yv[(p - 1) * N + k] : h[k];
            float dn[N];                                 // (Q == 1: the update beside the cell, weights read once)
#pragma unroll
            for (int i = 0; i < N; ++i) {
                float wr[ROWP];
#pragma unroll
                for (int k = 0; k < ROWP / 4; ++k) {
                    const float4 v = REG ? wreg[REG ? i * ROWP / 4 + k : 0] : reinterpret_cast<const float4 *>(sw)[i * ROWP / 4 + k];
                    wr[4 * k] = v.x; wr[4 * k + 1] = v.y; wr[4 * k + 2] = v.z; wr[4 * k + 3] = v.w;
                }
#pragma unroll
                for (int p = 0; p < Q; ++p) {
                    float ar = wr[3 * N + 3 * M], az = wr[3 * N + 3 * M + 1], aq = wr[3 * N + 3 * M + 2], an = wr[3 * N + 3 * M + 3];
                    if constexpr (M > 0) {
#pragma unroll
                        for (int k = 0; k < M; ++k) {
                            ar = fmaf(wr[3 * N + k], xv[p * XW + k], ar);
                            az = fmaf(wr[3 * N + M + k], xv[p * XW + k], az);
                            an = fmaf(wr[3 * N + 2 * M + k], xv[p * XW + k], an);
                        }
                    } else {
                        ar += xv[p * XW + i]; az += xv[p * XW + N + i]; an += xv[p * XW + 2 * N + i];
                    }
                    float ur = 0.0f, uz = 0.0f, un = 0.0f;
#pragma unroll
                    for (int k = 0; k < N; ++k) {
                        ar = fmaf(wr[k], hq[p][k], ar);
                        az = fmaf(wr[N + k], hq[p][k], az);
                        aq = fmaf(wr[2 * N + k], hq[p][k], aq);
                        if constexpr (Q == 1) {
                            ur = fmaf(wr[k], d[k], ur);
                            uz = fmaf(wr[N + k], d[k], uz);
                            un = fmaf(wr[2 * N + k], d[k], un);
                        }
                    }
                    const float r = rcp_approx(1.0f + ex2_approx(-LOG2E * ar)), z = rcp_approx(1.0f + ex2_approx(-LOG2E * az));
                    const float cc = fmaf(rcp_approx(1.0f + ex2_approx(2.0f * LOG2E * fmaf(r, aq, an))), -2.0f, 1.0f);         // tanh
                    const float omz = 1.0f - z, hc = hq[p][i] - cc;
                    const float kn = omz * fmaf(-cc, cc, 1.0f) * r, kr = kn * aq * (1.0f - r), kz = z * omz * hc, f = fmaf(z, hc, cc);
                    if constexpr (Q == 1) {
                        dn[i] = fmaf(z, d[i], fmaf(kr, ur, fmaf(kz, uz, fmaf(kn, un, f))));
                    } else {
                        cz[p][i] = z; ckr[p][i] = kr; ckz[p][i] = kz; ckn[p][i] = kn; cf[p][i] = f;
                    }
                }
            }
            // the updates, one position after the other
#pragma unroll
            for (int p = 0; p < Q; ++p) {
                const bool act = t0 + p >= 0 && t0 + p < te;
                if constexpr (Q > 1) {
#pragma unroll
                    for (int i = 0; i < N; ++i) {
                        float ur = 0.0f, uz = 0.0f, un = 0.0f;
                        float wr[3 * N];
#pragma unroll
                        for (int k = 0; k < (3 * N + 3) / 4; ++k) {
                            const float4 v = REG ? wreg[REG ? i * ROWP / 4 + k : 0] : reinterpret_cast<const float4 *>(sw)[i * ROWP / 4 + k];
                            if (4 * k < 3 * N) wr[4 * k] = v.x;
                            if (4 * k + 1 < 3 * N) wr[4 * k + 1] = v.y;
                            if (4 * k + 2 < 3 * N) wr[4 * k + 2] = v.z;
                            if (4 * k + 3 < 3 * N) wr[4 * k + 3] = v.w;
                        }
#pragma unroll
                        for (int k = 0; k < N; ++k) {
                            ur = fmaf(wr[k], d[k], ur);
                            uz = fmaf(wr[N + k], d[k], uz);
                            un = fmaf(wr[2 * N + k], d[k], un);
                        }
                        dn[i] = fmaf(cz[p][i], d[i], fmaf(ckr[p][i], ur, fmaf(ckz[p][i], uz, fmaf(ckn[p][i], un, cf[p][i]))));
                    }
                }
#pragma unroll
                for (int i = 0; i < N; ++i) {            // dn: the new iterate
                    const float v = dn[i] - yv[p * N + i];
                    if (own && act && i < n) mb = max(mb, __float_as_uint(fabsf(v)));
                    if (act) { d[i] = v; h[i] = yv[p * N + i]; yv[p * N + i] = dn[i]; }
                }
            }
            if constexpr (Q * N % 4 == 0) {
#pragma unroll
                for (int k = 0; k < Q * N / 4; ++k)
                    *reinterpret_cast<float4 *>(sy + i0 * N + 4 * k) = make_float4(yv[4 * k], yv[4 * k + 1], yv[4 * k + 2], yv[4 * k + 3]);
            }
        }
        __syncwarp();
        if (W * w >= burn) put(w);
        __syncwarp();
    }
    cp_async_wait_0();

    // ---- boundaries: this chain's end state against what its successor assumed
    unsigned mis = 0u;
    const long long wg = (long long)blockIdx.x * C::WARPS + warp;
    const bool prev = te > 0 && c > 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const float sn = __shfl_down_sync(0xffffffffu, start[k], 1);
        if (next && lane < 31) mis = max(mis, absdiff_bits(sn, d[k]));
    }
    const bool has_next = __shfl_sync(0xffffffffu, (int)next, 31) != 0, has_prev = __shfl_sync(0xffffffffu, (int)prev, 0) != 0 && wg > 0;
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {               // 0: behind this warp's chains (lane 31), 1: before them (lane 0)
        if (side == 0 ? !has_next : !has_prev) continue;
        const size_t edge = (size_t)hd.first_edge + (size_t)wg - side;
        float *slot = a.edge + edge * 2 * n;
        unsigned old = 0u;
        if (lane == (side == 0 ? 31 : 0)) {
#pragma unroll
            for (int k = 0; k < N; ++k) if (k < n) __stcg(slot + side * n + k, side == 0 ? d[k] : start[k]);
            __threadfence();
            old = atomicAdd(a.edge_flag + edge, 1u);
            if (old == 1u) {
                __threadfence();
#pragma unroll
                for (int k = 0; k < N; ++k) if (k < n) mis = max(mis, absdiff_bits(side == 0 ? d[k] : start[k], __ldcg(slot + (side ^ 1) * n + k)));
                a.edge_flag[edge] = 0u;
            }
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
        const unsigned prevc = atomicAdd(&st->exit_counter, 1u);
        if (prevc + 1u == nctas) {
            __threadfence();
            st->exit_counter = 0u;
            body_decide(st, a, W, BODY_ROUNDING);
        }
    }
}

}  // namespace deer
