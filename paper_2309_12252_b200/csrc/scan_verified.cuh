// The linear recurrence y_t = J_t y_{t-1} + b_t (Eq. 10; either direction) without matrix products: chains that start `burn`
// positions early from zero, each a plain sequence of matrix-vector steps, J read once (and a burn-in's worth of it twice).
// What a chain's start lacks is the state entering its burn-in, carried through `burn` Jacobians; that this vanished is
// verified: every chain's end state is compared with the start its successor assumed.  One boundary that differs by more than
// eta leaves StatusBlock::done at 0, and the chunked scan enqueued behind this launch (which multiplies the matrices out,
// Eq. 9) does the work; otherwise it returns at once.
// A state's components may have units of their own, and the chunked scan is good to fp32 in each: a component's difference is
// held to eta of that component's largest value over the VSCAN_WINDOW positions before the boundary (one position alone may be
// a zero crossing; more would measure a decayed value by what it decayed from) or of the sum of |terms| that its next value is
// made of, whichever is more -- what large components feed into a small one, no fp32 sum resolves better -- and to eta of the
// states' largest component.  (Without the terms, the gradient's scans of a GRU, lambda's components unequal, were done again:
// n = 64, B = 8, T = 2179, a training step 2.79 ms instead of 2.23.)
//
// G lanes per chain (n up to 32, a warp for n = 64); a matrix is read as consecutive 16-byte pieces: lane (sub, q) holds the
// columns 4q .. 4q+3 of the rows RP k + sub.  The next U positions' matrices are on their way in registers.
// What bounds it: HBM.  n = 8, B = 16, T = 2e5 (0.92 GB): 405 us by the chunked scan, which reads J twice and multiplies 8 x 8
// matrices at every position; floor 143 us.
#pragma once
#include "scan_onepass.cuh"

namespace deer {

template <int N> struct VScan {
    static constexpr int CQ = N / 4;                     // column quads
    static constexpr int G = N < 32 ? N : 32;            // lanes of a chain
    static constexpr int RP = G / CQ;                    // rows a load covers
    static constexpr int K = N / RP;                     // loads per position and lane
    static constexpr int OWN = N / G;                    // rows a lane owns: 4 q + sub (+ 2 e)
    static constexpr int U = N == 4 ? 16 : N == 8 ? 8 : N == 16 ? 4 : N == 32 ? 2 : 1;       // positions in flight
    static constexpr int CPW = 32 / G, WARPS = 4;
};

constexpr int VSCAN_WINDOW = 16;                         // (shorter than any burn-in and any chain)

struct VScanArgs {
    const float *J, *b, *y0;
    float *y;
    int B, T, L, burn;
    float eta;
    StatusBlock *st;
    float *edge;             // [chains][3][n]  end of the chain before, start and scale of the one behind
    unsigned *edge_flag;     // [chains]
};

__device__ __forceinline__ float4 ld_stream(const float4 *p)
{
    float4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

template <int N, bool REV>
__global__ void __launch_bounds__(128) scan_verified_kernel(VScanArgs a)
{
    using C = VScan<N>;
    constexpr int CQ = C::CQ, G = C::G, RP = C::RP, K = C::K, OWN = C::OWN, U = C::U, NN = N * N;
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cl = lane % G, sub = cl / CQ, q = cl % CQ, base = lane - cl;
    const int T = a.T, L = a.L, nchain = (T + L - 1) / L;
    const long long total = (long long)a.B * nchain;
    const long long gid0 = ((long long)blockIdx.x * C::WARPS + warp) * C::CPW + lane / G;
    const bool live = gid0 < total;
    const long long gid = live ? gid0 : total - 1;
    const long long seq = gid / nchain;
    const int c = (int)(gid - seq * nchain);
    const int own = c * L, first = max(0, own - a.burn), last = min(T, own + L);     // scan positions
    const float *Jseq = a.J + (size_t)seq * T * NN, *bseq = a.b + (size_t)seq * T * N;
    float *yseq = a.y + (size_t)seq * T * N;
    int row[OWN];
#pragma unroll
    for (int e = 0; e < OWN; ++e) row[e] = 4 * q + 2 * e + sub;

    // matrix and vector of scan position s (clamped: what lies outside is not used)
    float4 Jb[U][K];
    float bb[U][OWN];
    auto fetch = [&](int s, float4 (&M)[K], float (&v)[OWN]) {
        const int sc = min(s, last - 1);
        const int t = REV ? T - 1 - sc : sc, tm = REV ? min(t + 1, T - 1) : t;
        const float4 *src = reinterpret_cast<const float4 *>(Jseq + (size_t)tm * NN) + cl;
#pragma unroll
        for (int k = 0; k < K; ++k) M[k] = ld_stream(src + k * G);
#pragma unroll
        for (int e = 0; e < OWN; ++e) v[e] = __ldg(bseq + (size_t)t * N + row[e]);
    };
    float y[OWN];                                        // the lane's rows of the state
#pragma unroll
    for (int e = 0; e < OWN; ++e) y[e] = c == 0 && a.y0 ? a.y0[(size_t)seq * N + row[e]] : 0.0f;
    float start[OWN], scale[OWN];                        // scale: largest |y| of the last VSCAN_WINDOW positions before the own ones, or |terms|
#pragma unroll
    for (int e = 0; e < OWN; ++e) { start[e] = y[e]; scale[e] = 0.0f; }
#pragma unroll
    for (int u = 0; u < U; ++u) fetch(first + u, Jb[u], bb[u]);

    // z = M v (REV: M^T v), this lane's rows
    auto apply = [&](const float4 (&M)[K], const float (&v)[OWN], float (&z)[OWN]) {
        if constexpr (!REV) {
            // the four state entries of this lane's columns, then partial products, summed and scattered over the q lanes
            float yq[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                yq[k] = OWN == 1 ? __shfl_sync(FULL, v[0], base + k * CQ + q) : __shfl_sync(FULL, v[OWN == 1 ? 0 : k >> 1], base + (k & 1) * CQ + q);
            float part[K];
#pragma unroll
            for (int k = 0; k < K; ++k)
                part[k] = fmaf(M[k].x, yq[0], M[k].y * yq[1]) + fmaf(M[k].z, yq[2], M[k].w * yq[3]);
#pragma unroll
            for (int half = K / 2, mask = CQ / 2; mask > 0; half >>= 1, mask >>= 1) {
                const bool up = (q & mask) != 0;
#pragma unroll
                for (int k = 0; k < half; ++k) {
                    const float give = up ? part[k] : part[k + half], keep = up ? part[k + half] : part[k];
                    part[k] = keep + __shfl_xor_sync(FULL, give, mask);
                }
            }
#pragma unroll
            for (int e = 0; e < OWN; ++e) z[e] = part[e];
        } else {
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const float yk = __shfl_sync(FULL, v[OWN == 1 ? 0 : (k & 1)], base + sub * CQ + (OWN == 1 ? k : k >> 1));
                acc[0] = fmaf(M[k].x, yk, acc[0]); acc[1] = fmaf(M[k].y, yk, acc[1]);
                acc[2] = fmaf(M[k].z, yk, acc[2]); acc[3] = fmaf(M[k].w, yk, acc[3]);
            }
            if constexpr (RP == 4) {                 // sum and scatter over the four sub lanes
                const bool up2 = (sub & 2) != 0, up1 = (sub & 1) != 0;
                const float a0 = (up2 ? acc[2] : acc[0]) + __shfl_xor_sync(FULL, up2 ? acc[0] : acc[2], 2 * CQ);
                const float a1 = (up2 ? acc[3] : acc[1]) + __shfl_xor_sync(FULL, up2 ? acc[1] : acc[3], 2 * CQ);
                z[0] = (up1 ? a1 : a0) + __shfl_xor_sync(FULL, up1 ? a0 : a1, CQ);
            } else {
                const bool up1 = (sub & 1) != 0;
#pragma unroll
                for (int e = 0; e < OWN; ++e)
                    z[e] = (up1 ? acc[2 * e + 1] : acc[2 * e]) + __shfl_xor_sync(FULL, up1 ? acc[2 * e] : acc[2 * e + 1], CQ);
            }
        }
    };
    const int steps = __reduce_max_sync(FULL, last - first);
#pragma unroll 1
    for (int s0 = 0; s0 < steps; s0 += U) {
        if (s0 == a.burn) {                              // (the first own position of every chain that has a burn-in)
            float4 M[K];
            float v[OWN], z[OWN];
#pragma unroll
            for (int k = 0; k < K; ++k) M[k] = make_float4(fabsf(Jb[0][k].x), fabsf(Jb[0][k].y), fabsf(Jb[0][k].z), fabsf(Jb[0][k].w));
#pragma unroll
            for (int e = 0; e < OWN; ++e) v[e] = fabsf(y[e]);
            apply(M, v, z);
#pragma unroll
            for (int e = 0; e < OWN; ++e) scale[e] = fmaxf(scale[e], z[e] + fabsf(bb[0][e]));
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int s = first + s0 + u;
            if (s == own) {
#pragma unroll
                for (int e = 0; e < OWN; ++e) start[e] = y[e];
            }
            float z[OWN];
            apply(Jb[u], y, z);
            if (REV && s == 0) {
#pragma unroll
                for (int e = 0; e < OWN; ++e) z[e] = y[e];                           // (the first matrix of a reverse scan is the identity)
            }
            const bool in = s < last;
#pragma unroll
            for (int e = 0; e < OWN; ++e) {
                y[e] = in ? z[e] + bb[u][e] : y[e];
                if (s < own) scale[e] = fmaxf(s == own - VSCAN_WINDOW ? 0.0f : scale[e], fabsf(y[e]));
                if (in && s >= own && live) yseq[(size_t)(REV ? T - 1 - s : s) * N + row[e]] = y[e];
            }
            fetch(s + U, Jb[u], bb[u]);
        }
    }
    // ---- boundaries
    __shared__ unsigned bad;
    if (threadIdx.x == 0) bad = 0u;
    __syncthreads();
#pragma unroll
    for (int side = 0; side < 2; ++side) {               // 0: behind this chain, 1: before it
        const bool there = live && (side == 0 ? c + 1 < nchain : c > 0);
        const size_t edge = (size_t)(gid - side) ;
        float *slot = a.edge + edge * 3 * N;
        if (there) {
#pragma unroll
            for (int e = 0; e < OWN; ++e) {
                __stcg(slot + side * N + row[e], side == 0 ? y[e] : start[e]);
                if (side == 1) __stcg(slot + 2 * N + row[e], scale[e]);
            }
            __threadfence();
        }
        __syncwarp();
        unsigned old = 0u;
        if (there && cl == 0) { __threadfence(); old = atomicAdd(a.edge_flag + edge, 1u); }
        old = __shfl_sync(FULL, old, base);
        float diff = 0.0f, size = 0.0f;
        bool off = false;
        if (there && old == 1u) {
            __threadfence();
#pragma unroll
            for (int e = 0; e < OWN; ++e) {
                const float mine = side == 0 ? y[e] : start[e], other = __ldcg(slot + (side ^ 1) * N + row[e]);
                const float dv = fabsf(mine - other), sc = side == 0 ? __ldcg(slot + 2 * N + row[e]) : scale[e];
                off = off || !(dv <= a.eta * sc);        // (a NaN too)
                diff = fmaxf(diff, dv);
                size = fmaxf(size, fmaxf(fabsf(mine), fabsf(other)));
            }
            if (cl == 0) a.edge_flag[edge] = 0u;
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) {
            diff = fmaxf(diff, __shfl_xor_sync(FULL, diff, o));
            size = fmaxf(size, __shfl_xor_sync(FULL, size, o));
        }
        if (off || diff > a.eta * size) bad = 1u;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (bad) atomicOr(&a.st->mis_bits, 1u);
        __threadfence();
        const unsigned prev = atomicAdd(&a.st->exit_counter, 1u);
        if (prev + 1u == gridDim.x) {
            __threadfence();
            a.st->exit_counter = 0u;
            if (atomicExch(&a.st->mis_bits, 0u) == 0u) a.st->done = 1;
        }
    }
}

}  // namespace deer
