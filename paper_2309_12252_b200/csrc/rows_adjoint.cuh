// The whole gradient of a small cell (n, m in {1, 2, 4, 8}) in one launch: the adjoint solve of newton_adjoint.cuh (chains in
// descending time with a burn-in and verified boundaries, mu_t = J_{t+1}^T lambda_{t+1} as the state; see there) with n lanes
// per chain, one state component each, and the parameter gradients, dx and dy0 on the way.
//
// Lane i has row i of every weight matrix in registers: gates and p = (p_r, p_z, p_n) of its component, then its share
// sum_g W_g[i][j] p_g of every J^T lambda component j, summed and scattered over the chain's lanes by log2 n exchanges.  Its
// p times y_{t-1} and x are its rows of dW_h and dW_i: accumulated in registers over the chain, then over the CTA in a fixed
// order (slice b of the two-stage reduction; wgrad_final2_kernel adds the slices).  The inputs of the next U positions are
// requested ahead; no Jacobian, lambda or pre-activation gradient is ever stored.
// What bounds it: issue slots (about 170 per step and warp, 95 in the burn-in; 55 % used at n = 8, m = 4, B = 16, T = 1e4) and
// the latency that 11 warps per SM leave.  Before: a cell that wrote Jacobians, a scan
// that read them, a VJP pass: n = 8, m = 4, B = 16, T = 1e4 92 us, n = m = 8, T = 1e6 6.1 ms.
#pragma once
#include <type_traits>
#include "newton_adjoint.cuh"

namespace deer {

template <int N, int M> struct RowsAdj {
    static constexpr int THREADS = 128, G = THREADS / N; // chains of a CTA
    static constexpr int VI = 3 * (M + 1), VALS = VI + 3 * (N + 1);
    static constexpr int U = N == 8 || M == 8 ? 2 : 4;   // positions requested ahead
    static constexpr int CTAS = N + M > 8 ? 3 : 4;       // (registers)
};

// v[0 .. K) summed over the LANES lanes of a group (a power of two) and scattered: lane l keeps max(K / LANES, 1) sums in
// v[0 ..), those of k = l * K / LANES + .. (K < LANES: of k = l * K / LANES).
template <int K, int LANES>
__device__ __forceinline__ void reduce_scatter(float (&v)[K], int l)
{
    int have = K;
#pragma unroll
    for (int mask = LANES / 2; mask > 0; mask >>= 1) {
        if (have > 1) {
            have >>= 1;
            const bool up = (l & mask) != 0;
#pragma unroll
            for (int k = 0; k < K / 2; ++k)
                if (k < have) {
                    const float give = up ? v[k] : v[k + have], keep = up ? v[k + have] : v[k];
                    v[k] = keep + __shfl_xor_sync(0xffffffffu, give, mask);
                }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], mask);
        }
    }
}

struct RowsAdjOut { float *partial_i, *partial_h, *dx; };

template <int N, int M>
__global__ void __launch_bounds__(128, (RowsAdj<N, M>::CTAS)) rows_adjoint_kernel(AdjArgs a, RowsAdjOut out)
{
    using C = RowsAdj<N, M>;
    constexpr int U = C::U, VI = C::VI, VALS = C::VALS;
    constexpr float LOG2E = 1.4426950408889634f;
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ float red[4][N][VALS + 1];
    StatusBlock *st = a.st;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, i = lane % N;
    const int L = a.L, T = a.T, burn = a.burn, nchain = (T + L - 1) / L;
    if (*(volatile int *)&st->done) return;

    float wr[N], wz[N], wn[N], vr[M], vz[M], vn[M];
#pragma unroll
    for (int k = 0; k < N; ++k) { wr[k] = a.h0.W_h[i * N + k]; wz[k] = a.h0.W_h[(N + i) * N + k]; wn[k] = a.h0.W_h[(2 * N + i) * N + k]; }
#pragma unroll
    for (int k = 0; k < M; ++k) { vr[k] = a.h0.W_i[i * M + k]; vz[k] = a.h0.W_i[(N + i) * M + k]; vn[k] = a.h0.W_i[(2 * N + i) * M + k]; }
    const float br = a.h0.b_h[i] + a.h0.b_i[i], bz = a.h0.b_h[N + i] + a.h0.b_i[N + i], bq = a.h0.b_h[2 * N + i], bn = a.h0.b_i[2 * N + i];

    const long long total = (long long)a.B * nchain, gid = (long long)blockIdx.x * C::G + tid / N;
    const long long b = gid < total ? gid / nchain : 0;
    const int c = gid < total ? (int)(gid - b * nchain) : 0;
    const int te = gid < total ? min(T, (c + 1) * L) : 0, ts = c * L - burn;       // scan positions: q is time step T - 1 - q
    const bool next = te > 0 && (c + 1) * L < T, prev = te > 0 && c > 0;
    const float *yb = a.y + (size_t)b * T * N, *gb = a.gy + (size_t)b * T * N, *xb = a.x + (size_t)b * T * M, *y0 = a.y0 + (size_t)b * N;

    float hb[U][N], xv[U][M], gv[U];
    auto fetch = [&](int q, float (&h)[N], float (&x)[M], float &g) {              // (clamped: what lies outside is not used)
        const int t = T - 1 - min(max(q, 0), T - 1);
        const float *hp = t > 0 ? yb + (size_t)(t - 1) * N : y0, *xp = xb + (size_t)t * M;
        if constexpr (N >= 4) {
#pragma unroll
            for (int k = 0; k < N / 4; ++k) {
                const float4 v = __ldg(reinterpret_cast<const float4 *>(hp) + k);
                h[4 * k] = v.x; h[4 * k + 1] = v.y; h[4 * k + 2] = v.z; h[4 * k + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < N; ++k) h[k] = __ldg(hp + k);
        }
#pragma unroll
        for (int k = 0; k < M; ++k) x[k] = __ldg(xp + k);
        g = __ldg(gb + (size_t)t * N + i);
    };
    float mu = 0.0f, start = 0.0f, scale = 0.0f;         // scale: of the boundary before this chain
    unsigned mb = 0u;
    float ai[3][M + 1], ah[3][N + 1];
#pragma unroll
    for (int g = 0; g < 3; ++g) {
#pragma unroll
        for (int k = 0; k <= M; ++k) ai[g][k] = 0.0f;
#pragma unroll
        for (int k = 0; k <= N; ++k) ah[g][k] = 0.0f;
    }
    auto step = [&](int s, int u, auto own) {
        constexpr bool OWN = decltype(own)::value;
        const int q = ts + s;
        const bool act = q >= 0 && q < te;
        float ar = br, az = bz, aq = bq, an = bn, h = 0.0f;
#pragma unroll
        for (int k = 0; k < M; ++k) { ar = fmaf(vr[k], xv[u][k], ar); az = fmaf(vz[k], xv[u][k], az); an = fmaf(vn[k], xv[u][k], an); }
#pragma unroll
        for (int k = 0; k < N; ++k) {
            ar = fmaf(wr[k], hb[u][k], ar); az = fmaf(wz[k], hb[u][k], az); aq = fmaf(wn[k], hb[u][k], aq);
            if (k == i) h = hb[u][k];
        }
        const float r = rcp_approx(1.0f + ex2_approx(-LOG2E * ar)), z = rcp_approx(1.0f + ex2_approx(-LOG2E * az));
        const float cc = fmaf(rcp_approx(1.0f + ex2_approx(2.0f * LOG2E * fmaf(r, aq, an))), -2.0f, 1.0f);       // tanh
        const float lam = gv[u] + mu, lo = (1.0f - z) * lam;
        if (act) mb = max(mb, __float_as_uint(fabsf(lam)));
        float pz = lo * z * (h - cc), pa = lo * fmaf(-cc, cc, 1.0f), pn = pa * r, pr = pn * aq * (1.0f - r);
        float sh[N];
#pragma unroll
        for (int k = 0; k < N; ++k) sh[k] = fmaf(wr[k], pr, fmaf(wz[k], pz, wn[k] * pn));
        reduce_scatter<N, N>(sh, i);
        if constexpr (OWN) {
            if (!act) { pr = 0.0f; pz = 0.0f; pn = 0.0f; pa = 0.0f; }
#pragma unroll
            for (int k = 0; k < M; ++k) { ai[0][k] = fmaf(pr, xv[u][k], ai[0][k]); ai[1][k] = fmaf(pz, xv[u][k], ai[1][k]); ai[2][k] = fmaf(pa, xv[u][k], ai[2][k]); }
#pragma unroll
            for (int k = 0; k < N; ++k) { ah[0][k] = fmaf(pr, hb[u][k], ah[0][k]); ah[1][k] = fmaf(pz, hb[u][k], ah[1][k]); ah[2][k] = fmaf(pn, hb[u][k], ah[2][k]); }
            ai[0][M] += pr; ai[1][M] += pz; ai[2][M] += pa; ah[2][N] += pn;         // (db_h of r and z: db_i's)
            if (out.dx) {
                float dxv[M];
#pragma unroll
                for (int k = 0; k < M; ++k) dxv[k] = fmaf(vr[k], pr, fmaf(vz[k], pz, vn[k] * pa));
                reduce_scatter<M, N>(dxv, i);
                constexpr int KEEP = M > N ? M / N : 1;
                float *o = out.dx + ((size_t)b * T + (T - 1 - min(max(q, 0), T - 1))) * M;
                if (act && (M >= N || i % (N / (M < N ? M : N)) == 0)) {
#pragma unroll
                    for (int k = 0; k < KEEP; ++k) o[(M >= N ? i * KEEP : i / (N / (M < N ? M : N))) + k] = dxv[k];
                }
            }
        }
        mu = act ? fmaf(z, lam, sh[0]) : mu;
    };
    using No = std::false_type;
    using Yes = std::true_type;
    // (every chain of the launch has the same number of steps: burn and L are multiples of U)
    const int s0 = nchain == 1 ? burn : 0, s_end = burn + min(L, (T + U - 1) / U * U);
    const bool live = __any_sync(FULL, te > 0);
    if (live) {
#pragma unroll
        for (int u = 0; u < U; ++u) fetch(ts + s0 + u, hb[u], xv[u], gv[u]);
#pragma unroll 1
        for (int s = s0; s < burn; s += U) {
            if (s == burn - ADJ_WINDOW) mb = 0u;
#pragma unroll
            for (int u = 0; u < U; ++u) { step(s + u, u, No{}); fetch(ts + s + U + u, hb[u], xv[u], gv[u]); }
        }
        start = mu;
        unsigned top = mb;
#pragma unroll
        for (int o = N / 2; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(FULL, top, o));
        scale = __uint_as_float(top);
#pragma unroll 1
        for (int s = burn; s < s_end; s += U) {
#pragma unroll
            for (int u = 0; u < U; ++u) { step(s + u, u, Yes{}); fetch(ts + s + U + u, hb[u], xv[u], gv[u]); }
        }
    }
    // ---- this CTA's slice of the parameter gradients: lanes of equal i over the warp, then the warps in order
    auto warp_sum = [&](float v) {
#pragma unroll
        for (int o = 16; o >= N; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
        return v;
    };
#pragma unroll
    for (int g = 0; g < 3; ++g) {
#pragma unroll
        for (int k = 0; k <= M; ++k) { const float v = warp_sum(ai[g][k]); if (lane < N) red[warp][i][g * (M + 1) + k] = v; }
#pragma unroll
        for (int k = 0; k <= N; ++k) { const float v = warp_sum(k == N && g < 2 ? ai[g][M] : ah[g][k]); if (lane < N) red[warp][i][VI + g * (N + 1) + k] = v; }
    }
    __syncthreads();
    for (int o = tid; o < N * VALS; o += C::THREADS) {
        const int row = o / VALS, v = o % VALS;
        const float sum = ((red[0][row][v] + red[1][row][v]) + red[2][row][v]) + red[3][row][v];
        if (v < VI) out.partial_i[(size_t)blockIdx.x * (3 * N * (M + 1)) + ((v / (M + 1)) * N + row) * (M + 1) + v % (M + 1)] = sum;
        else out.partial_h[(size_t)blockIdx.x * (3 * N * (N + 1)) + (((v - VI) / (N + 1)) * N + row) * (N + 1) + (v - VI) % (N + 1)] = sum;
    }
    // ---- the gradient w.r.t. y0, and the boundaries
    unsigned mb_end = 0u, mis = 0u, rel = 0u, mis_end = 0u;
    if (te > 0 && !next) {
        if (a.dy0) a.dy0[(size_t)b * N + i] = mu;
        mb_end = __float_as_uint(fabsf(mu));             // (wanted or not: see adjoint_decide)
    }
    const int reach = DY0_REACH * burn;
    if constexpr (N < 32) {                              // the next chain of this warp
        const float sn = __shfl_down_sync(FULL, start, N), sc = __shfl_down_sync(FULL, scale, N);
        if (next && lane + N < 32) {
            mis = absdiff_bits(sn, mu);
            rel = boundary_ratio(mis, sc);
            if (T - te < reach) mis_end = mis;
        }
    }
    const long long wg = (long long)blockIdx.x * 4 + warp;
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {               // 0: behind this warp's chains, 1: before them
        const bool mine = side == 0 ? lane >= 32 - N && next : lane < N && prev && wg > 0;
        const size_t edge = (size_t)(wg - side);
        float *slot = a.edge + edge * ADJ_EDGE(N);
        if (mine) {
            __stcg(slot + side * N + i, side == 0 ? mu : start);
            if (side == 1 && i == 0) __stcg(slot + 2 * N, scale);
            __threadfence();
        }
        __syncwarp();
        unsigned old = 0u;
        const int leader = side == 0 ? 32 - N : 0;
        if (mine && lane == leader) { __threadfence(); old = atomicAdd(a.edge_flag + edge, 1u); }
        old = __shfl_sync(FULL, old, leader);
        if (mine && old == 1u) {
            __threadfence();
            const unsigned q = absdiff_bits(side == 0 ? mu : start, __ldcg(slot + (side ^ 1) * N + i));
            mis = max(mis, q);
            rel = max(rel, boundary_ratio(q, side == 0 ? __ldcg(slot + 2 * N) : scale));
            if (T - (side == 0 ? te : c * L) < reach) mis_end = max(mis_end, q);
            if (lane == leader) a.edge_flag[edge] = 0u;
        }
    }
    mb = __reduce_max_sync(FULL, mb);
    mis = __reduce_max_sync(FULL, mis);
    rel = __reduce_max_sync(FULL, rel);
    mb_end = __reduce_max_sync(FULL, mb_end);
    mis_end = __reduce_max_sync(FULL, mis_end);
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
        const unsigned prevc = atomicAdd(&st->exit_counter, 1u);
        if (prevc + 1u == gridDim.x) {
            __threadfence();
            st->exit_counter = 0u;
            adjoint_decide(st, a.eta, a.dy0 != nullptr, burn);
        }
    }
}

}  // namespace deer
