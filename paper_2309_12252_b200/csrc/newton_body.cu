// Launch side of the one-launch Newton body.
#include <math.h>
#include <algorithm>
#include <mutex>
#include <stdlib.h>
#include "newton_body.h"

namespace deer {

BodyKernels body_kernels_8(bool, bool);
BodyKernels body_kernels_16(bool, bool);
BodyKernels body_kernels_24(bool, bool);
BodyKernels body_kernels_32(bool, bool);
BodyKernels body_kernels_40(bool, bool);
BodyKernels body_kernels_48(bool, bool);
BodyKernels body_kernels_56(bool, bool);
BodyKernels body_kernels_64(bool, bool);

// n = 16, 32, 64: sizes whose linear solve has always run in reduced precision (bf16 / single-TF32 chain products)
static bool reduced(int n) { return n == 16 || n == 32 || n == 64; }

// A kernel per state size (rounded up to a multiple of 8) and row alignment.
static BodyKernels pick(int n, bool v2)
{
    const bool exact = !reduced(n);
    switch ((n + 7) / 8) {
    case 1: return body_kernels_8(v2, exact);
    case 2: return body_kernels_16(v2, exact);
    case 3: return body_kernels_24(v2, exact);
    case 4: return body_kernels_32(v2, exact);
    case 5: return body_kernels_40(v2, exact);
    case 6: return body_kernels_48(v2, exact);
    case 7: return body_kernels_56(v2, exact);
    default: return body_kernels_64(v2, exact);
    }
}

constexpr size_t BODY_SMEM_MAX = 226 * 1024;          // (dynamic; the kernels have a few static words besides)

bool body_supported(int n, int m, bool have_u)
{
    if (n < 1 || n > 64) return false;
    return have_u || (m <= 64 && pick(n, false).one_smem((m + 7) / 8) <= BODY_SMEM_MAX);
}

// What a body's boundaries have to be good to, as a part of its update, and the burn-in that a cell as initialised needs for
// it (white-noise inputs).  Reduced-precision solves: a thousandth.  The others: fp32 level where the caller counts bodies
// (tol < 0), else 1e-4 -- the loop then ends on a body whose update is below tol, so the result is good to 1e-4 of that.
float body_eta(int n, float tol) { return reduced(n) ? 1e-3f : tol > 0.0f ? 1e-4f : 4e-6f; }
int body_first_burn(int n, float tol) { return reduced(n) ? 24 : tol > 0.0f ? 30 : 40; }

// Behind a zero guess the first update is of order one and its boundaries are asked for a twentieth of it: 16 or 24 steps, where
// a body's time goes with them.  (Rates seen at first bodies, per step: white noise 0.32 ... 0.44, random walks and sinusoids
// 0.12 ... 0.3; the twentieth takes 0.19 or 0.125.)
int body_start_burn(int n, float tol, bool adapt) { return tol > 0.0f && adapt ? (reduced(n) ? 16 : 24) : body_first_burn(n, tol); }

// Shared-memory opt-in and CTAs per SM of a kernel, looked up once per kernel, device and shared-memory size.
static int occupancy_of(const void *kern, int threads, size_t smem)
{
    static std::mutex mu;
    struct Entry { const void *k; size_t smem; int dev, occ; };
    static Entry cache[128];
    static int used = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    for (int i = 0; i < used; ++i)
        if (cache[i].k == kern && cache[i].smem == smem && cache[i].dev == dev) return cache[i].occ;
    if (smem > 48 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BODY_SMEM_MAX);
    int o = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, threads, smem) != cudaSuccess || o < 1) o = 1;
    if (used < 128) cache[used++] = {kern, smem, dev, o};
    return o;
}

static int sm_count()
{
    static int sms[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    if (!sms[dev]) {
        int v = 0;
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        sms[dev] = v > 0 ? v : 148;
    }
    return sms[dev];
}

// CTAs of `per_cta` chains of length L: in all, of the head that needs most, and boundaries between units of `unit` chains.
struct Count { long long ctas, edges; int worst; };
static Count count_ctas(int B, int T, const int *strides, int H, int L, int per_cta, int unit)
{
    Count c{0, 0, 0};
    for (int h = 0; h < H; ++h) {
        const int s = strides ? strides[h] : 1, Tp = (T + s - 1) / s;
        const long long chains = (long long)B * s * ((Tp + L - 1) / L), k = (chains + per_cta - 1) / per_cta;
        c.ctas += k;
        c.edges += (chains + unit - 1) / unit;
        c.worst = (int)std::max<long long>(c.worst, k);
    }
    return c;
}

static int longest(int T, const int *strides, int H)
{
    int w = 1;
    for (int h = 0; h < H; ++h) w = std::max(w, (T + (strides ? strides[h] : 1) - 1) / (strides ? strides[h] : 1));
    return w;
}

// One-phase plans: the chain length with the least estimated time.  Every CTA runs its chains' steps (burn-in and L, or the
// whole sequence where it is no longer than L) and `cap` of them run at a time, so the launch takes the longest CTA's steps or
// the sum over CTAs / cap, whichever is more.  `alone`: time of a step of a nearly empty GPU as a part of a full one's (thread
// and warp chains: n = 1 0.57 us at 0.1 waves, 1.0 at 0.75; n = 8 1.5 at 0.3, 2.1 at 0.8; n = 16 2.8 at 0.5, 3.2 at 1); below
// zero: of a CTA that has half of its tiles, else the same throughout (n = 32 tiles: 3.5 us, 4.6 with both).
static void one_wave_of_chains(BodyPlan *p, const void *kern, int threads, int chains, int edge_unit, int gran, size_t smem, int burn, int B, int T, const int *strides, int H, float alone = 0.6f, int occ_cap = 64)
{
    const int Tmax = longest(T, strides, H);
    p->NC = 0;
    p->whole_loop = false;
    p->warps = threads / 32;
    p->smem = smem;
    const long long cap = (long long)sm_count() * std::min(occ_cap, occupancy_of(kern, threads, smem));      // CTAs of one wave
    p->share = (float)((double)B * T * H / ((double)cap * chains));
    double best = 0.0;
    // (gran: what the chain length is a multiple of)
    for (int L = std::max(CHAIN_L_MIN, gran); ; L += std::max(gran, L / 32 / gran * gran)) {
        double sum = 0.0, top = 0.0;
        for (int h = 0; h < H; ++h) {
            const int s = strides ? strides[h] : 1, Tp = (T + s - 1) / s, nch = (Tp + L - 1) / L;
            const double ctas = (double)(((long long)B * s * nch + chains - 1) / chains), steps = nch > 1 ? L + burn : Tp;
            sum += ctas * steps;
            top = std::max(top, steps);
        }
        // (a launch of a little more than one wave takes two: whole waves, as far as a few of them go)
        const double waves = sum / top / (double)cap, whole = waves <= 4.0 ? ceil(waves - 1e-9) : waves;
        const double cost = top * (waves >= 1.0 ? whole : alone < 0.0f ? (waves <= 0.5 ? -alone : 1.0) : alone + (1.0 - alone) * waves);
        if (best == 0.0 || cost < best) { best = cost; p->L = L; p->waves = (float)waves; }
        if (L >= Tmax || (best > 0.0 && fabsf(alone) * top > best)) break;
    }
    const Count c = count_ctas(B, T, strides, H, p->L, chains, edge_unit);
    p->max_ctas = c.worst; p->edges = c.edges;
}

// Burn-ins that are worth trying.  A launch takes burn + L steps, whatever its size while it is one wave; the kernels that
// multiply the Jacobians out take `a` such steps' time for a small problem and `b` for every position of `share` more (B200, us
// per body, here per step / there, positions in thousands, m = 4 or 8):
//   n = 1   0.6-1.0 / 34 (192) 44 (1,600)              n = 16  2.8-3.2 / 148 (240) 280 (640)
//   n = 2   0.6-0.8 / 32 (192) 66 (1,600)              n = 32  3.5-4.6 / 106 (32) 193 (128) 554 (640)
//   n = 4   0.75-0.9 / 39 (192) 120 (1,600)            n = 64  5.0-6.4 / 311 (16) 714 (128) 1508 (320)
//   n = 8   1.5-2.1 / 72 (192) 178 (640) 396 (1,600)
// Only the powers of two have tuned kernels of that kind; the others' are an order of magnitude slower.
// The two-launch scans of n >= 16 take as long for one sequence as for four (n = 32, B = 1, T = 6.4e4: 340 us per body).
static int worth_trying(const BodyPlan &p, int n, int m, int B)
{
    float a, b;
    const float share = n >= 16 && B < 4 ? p.share * 4.0f / (float)B : p.share;
    switch (n) {
    case 1: case 2: a = 45.0f; b = 2.0f; break;
    case 4: a = 30.0f; b = 2.7f; break;
    case 8: a = 24.0f; b = 4.0f; break;
    case 16: a = 30.0f; b = 2.6f; break;
    case 32: a = 2700.0f / (float)(128 + m); b = 1000.0f / (float)(128 + m); break;      // (a step of m = 32 takes 4.5 us)
    case 64: a = 36.0f; b = 13.0f; break;
    default: return std::max(320, 8 * p.L);
    }
    return (int)(a + b * share) - p.L;
}

bool body_plan(BodyPlan *p, BodyForm form, int B, int T, int n, int m, bool have_u, const int *strides, int H)
{
    const int kx = have_u ? 0 : (m + 7) / 8, sms = sm_count(), Tmax = longest(T, strides, H);
    if (form != BodyForm::TILE && form != BodyForm::LANE && !body_supported(n, m, have_u)) return false;
    const BodyKernels k = pick(n, (n & 1) == 0);
    p->form = form;
    if (form == BodyForm::LANE) {
        if (n > 8 || (!have_u && m > 8)) return false;
        const LaneKernel lk = lane_kernel(n, m, have_u);
        const int burn = (body_first_burn(n, 1.0f) + lk.W - 1) / lk.W * lk.W;
        one_wave_of_chains(p, (const void *)lk.kern, 128, 128, 32, lk.W, lk.smem, burn, B, T, strides, H);
        p->burn_cap = worth_trying(*p, n, m, B);
        return true;
    }
    if (form == BodyForm::TILE) {
        if (!(n == 32 || n == 64) || have_u || m > 64 || H != 1 || strides) return false;
        if (k.tile_smem(m) > BODY_SMEM_MAX) return false;
        one_wave_of_chains(p, (const void *)k.tile(m), k.tile_threads, k.tile_chains, 128, 1, k.tile_smem(m), body_first_burn(n, 1.0f), B, T, strides, H, n == 32 ? -0.75f : 1.0f);
        if (p->edges <= sms) p->max_ctas = (int)p->edges;      // (two tiles per CTA only where there are more than SMs)
        p->burn_cap = worth_trying(*p, n, m, B);
        return true;
    }
    if (form == BodyForm::TWO_PHASE) {
        const size_t fixed = k.seg_fixed(kx);
        if (fixed >= BODY_SMEM_MAX) return false;
        const int slots = (int)((BODY_SMEM_MAX - fixed) / k.slot_bytes);
        const int cap = std::min(96, slots / 2), own = slots - cap;
        if (own < 80) return false;
        p->warps = k.seg_warps;
        p->burn_cap = cap;
        // The shortest chains for which the problem is one wave of CTAs, one per SM: a body then takes burn + L short steps.
        // Where none is short enough, the CTA that holds most positions.
        for (int L = 5; ; L += 2) {
            const int nc_fit = std::min(k.nc_max, own / L / 16 * 16);
            if (nc_fit < 16) break;
            int NC = 16;
            while (2 * NC <= nc_fit && count_ctas(B, T, strides, H, L, NC, NC).ctas > sms) NC *= 2;
            const Count c = count_ctas(B, T, strides, H, L, NC, NC);
            if (p->NC * p->L < NC * L || c.ctas <= sms) {
                p->NC = NC; p->L = L; p->max_ctas = c.worst; p->edges = c.edges;
                p->waves = (float)c.ctas / (float)sms;
                p->smem = fixed + k.slot_bytes * (size_t)(cap + NC * L);
            }
            p->whole_loop = (long long)c.worst * H <= sms;      // (the grid is max_ctas x H)
            if (c.ctas <= sms || L >= Tmax) break;
        }
        if (!(p->NC > 0 && p->max_ctas > 0)) return false;
        // A step of a chain takes an eighth of a microsecond (n <= 8) to a half; a body of the other kernels 30 to 90 us.  The
        // slots that the CTA's own positions leave are there for longer burn-ins.
        p->burn_cap = std::max(cap, std::min(slots - p->NC * p->L, (n & (n - 1)) != 0 ? 512 : n <= 8 ? 128 : 224));
        p->smem = fixed + k.slot_bytes * (size_t)(p->burn_cap + p->NC * p->L);
        return true;
    }
    if (n <= 8) return false;
    one_wave_of_chains(p, (const void *)k.one, 32 * k.one_warps, 16 * k.one_warps, 16, 1, k.one_smem(kx), body_first_burn(n, 1.0f), B, T, strides, H);
    p->burn_cap = worth_trying(*p, n, m, B);
    return true;
}

bool adjoint_supported(int n, int m, bool have_u)
{
    if (n < 1 || n > 64) return false;
    return have_u || (m <= 64 && pick(n, false).adj_smem((m + 7) / 8) <= BODY_SMEM_MAX);
}

bool adjoint_plan(BodyPlan *p, int B, int T, int n, int m, bool have_u, const int *strides, int H)
{
    if (!adjoint_supported(n, m, have_u)) return false;
    const BodyKernels k = pick(n, (n & 1) == 0);
    if (k.adj_smem(have_u ? 0 : (m + 7) / 8) > BODY_SMEM_MAX) return false;
    one_wave_of_chains(p, (const void *)k.adj(have_u ? 0 : m), 32 * k.one_warps, 16 * k.one_warps, 16, 1, k.adj_smem(have_u ? 0 : (m + 7) / 8), ADJ_BURN, B, T, strides, H, 0.8f);
    return true;
}

size_t adjoint_starts(int n) { return n > 48 ? 16 * (size_t)((n + 7) / 8 * 8 + 4) : 0; }

// From how many positions on is the adjoint launch faster than the kernels that multiply the Jacobians out?  Its time is that
// of its steps (44 + 16 of them, some 3 us each, more with the channels that a step contracts) until the chains fill the GPU.
// (B200, us per gradient, here / there, B = 8: n = 9, m = 8 202 / 138 at 6,400 positions, 208 / 200 at 20,000; n = 20, m = 8
// 228 / 244 at 6,400; n = 28, m = 60 530 / 400 at 6,400, 561 / 737 at 20,000; n = 16, m = 3 219 / 180 at 80,000, 295 / 305 at
// 160,000; n = 32, B = 16, m = 3 295 / 251 at 48,000, 322 / 330 at 64,000, m = 32 374 / 309 at 64,000, 405 / 416 at 96,000, m = 64
// 494 / 443 at 96,000, 516 / 544 at 128,000;
// n = 64, here a tile, 728 / 525 at 20,000, 793 / 722 at 40,000, 819 / 881 at 56,000 whatever m.)
// n <= 4 pads to 8 columns where its own kernels are tuned; n = 64 with m > 64 is no tile's (nor worth its spills early).
static float adjoint_line(int n, int m)
{
    const float c = (float)m;
    switch (n) {
    case 1: case 2: case 4: return 1e30f;
    case 8: return 270000.0f;
    case 16: return 120000.0f * (1.0f + c / 20.0f);
    case 32: return 70000.0f * (1.0f + c / 55.0f);
    case 64: return m <= 64 ? 50000.0f : 250000.0f;
    }
    if (n < 8) return 4000.0f * (1.0f + c / 8.0f);
    if (n < 16) return 180000.0f / (float)n * (1.0f + c / 40.0f);
    return 4000.0f * (1.0f + c / 30.0f);
}

// The other kernels' time grows with the positions: at k times the line it is that of k (44 + 16) steps.
int adjoint_burn_cap(int n, int m, long long positions, int L)
{
    return (int)fminf(512.0f, (float)(ADJ_BURN + 16) * ((float)positions / adjoint_line(n, m))) - L;
}

int launch_newton_adjoint(const AdjArgs &a, const BodyPlan &p, cudaStream_t st)
{
    const bool aligned = (((uintptr_t)a.y | (uintptr_t)a.gy | (uintptr_t)a.y0 | (uintptr_t)a.u | (uintptr_t)a.lam | (uintptr_t)a.dGi |
                           (uintptr_t)a.dGh) & 7) == 0;
    const BodyKernels k = pick(a.n, (a.n & 1) == 0 && aligned);
    auto kern = k.adj(a.u ? 0 : a.m);
    occupancy_of((const void *)kern, 32 * p.warps, p.smem);
    DEER_KERNEL("newton_adjoint_kernel", st,
                kern<<<dim3((unsigned)p.max_ctas, (unsigned)a.H), 32 * p.warps, p.smem, st>>>(a));
    return DEER_OK;
}

bool rows_adjoint_plan(BodyPlan *p, int B, int T, int n, int m, int max_ctas)
{
    auto small = [](int v) { return v == 1 || v == 2 || v == 4 || v == 8; };
    if (!small(n) || !small(m)) return false;
    one_wave_of_chains(p, (const void *)rows_adjoint_of(n, m), 128, 128 / n, 32 / n, 4, 0, ADJ_BURN, B, T, nullptr, 1, 0.6f, std::max(1, max_ctas / sm_count()));
    return p->max_ctas <= max_ctas;
}

// (n = 32 gains nothing over sixteen chains per warp: 2270 / 2286 us at 1.6e6 positions.)
bool adjoint_tile_plan(BodyPlan *p, int B, int T, int n, int m)
{
    if (n != 64 || m > 64) return false;
    const BodyKernels k = pick(n, true);
    if (k.adj_tile_smem(m) > BODY_SMEM_MAX) return false;
    one_wave_of_chains(p, (const void *)k.adj_tile(m), k.tile_threads, k.tile_chains, 128, 1, k.adj_tile_smem(m), ADJ_BURN, B, T, nullptr, 1, 1.0f);
    return true;
}

int launch_adjoint_tile(const AdjArgs &a, const BodyPlan &p, cudaStream_t st)
{
    const BodyKernels k = pick(a.n, true);
    occupancy_of((const void *)k.adj_tile(a.m), 32 * p.warps, p.smem);
    DEER_KERNEL("adjoint_tile_kernel", st, k.adj_tile(a.m)<<<(unsigned)p.max_ctas, 32 * p.warps, p.smem, st>>>(a));
    return DEER_OK;
}

// Measured lines (B200, m = n unless stated, us per evaluation: two-phase / one-phase / multiplied-out kernels):
//   n = 4, B = 1, T = 1,000:   75 /  -  / 104      n = 4,  B = 16, T = 3e4: 591 / 354 / 188
//   n = 8, B = 16, T = 1e4 (m = 4): 129 / - / 231   n = 8,  B = 16, T = 3e4: 570 / 321 / 539   n = 8,  T = 1e5: 1733 / 704 / 1564
//   n = 16, B = 8, T = 2e4:   302 / 410 / 452      n = 16, B = 16, T = 1e5: 2407 / 1108 / 2283
//   n = 32, B = 16, T = 1e3:  128 / 887 / 353      n = 32, B = 16, T = 1e4: 876 / 1126 / 873
//   n = 64, B = 16, T = 1e3:    - / 2369 / 1247    n = 64, B = 16, T = 1e4:   - / 2828 / 3345
// Two-phase: one wave (then the whole loop is one launch), two waves from n = 9 on.  One-phase: from half a wave of chains on --
// below, its steps, a whole cell each, are a serial chain that nothing fills (n <= 8 never comes here: a thread per chain).
// Sizes without tuned kernels of the other kind always come here, to the two-phase kernel up to four, five or six waves: there random
// walks, whose bodies the long chains of the other run again, break even; white noise does so earlier (B = 16, m = 8, us per
// evaluation, two-phase / one-phase, white noise then random walks, the last before the line and the first behind it):
//   n = 12   T = 12,000 433 / 386, 669 / 893      T = 16,000 552 / 406, 1100 / 988
//   n = 20   T = 12,000 566 / 492, 875 / 969      T = 16,000 795 / 498, 1224 / 985
//   n = 24   T = 12,000 553 / 498, 663 / 759      T = 16,000 781 / 508, 1185 / 1001
//   n = 28   T = 8,000 614 / 545, 928 / 1012      T = 9,500 722 / 570, 1139 / 1136
//   n = 40   T = 4,000 652 / 714, 814 / 1076      T = 5,000 803 / 731, 1034 / 1171
//   n = 48   T = 3,200 774 / 896, 924 / 1270      T = 4,000 919 / 900, 1084 / 1235
// A thread per chain, powers of two: by positions per chain of a full GPU (`share`; m = n or 4, B = 16, white noise then random
// walks, where a try is often lost: thread per chain / multiplied out):
//   n = 1   13 175 / 208, 128 / 156   30 205 / 235, 141 / 174   42 217 / 302, 162 / 221   84 301 / 541, 226 / 411
//   n = 2   20 229 / 210, 363 / 306   26 268 / 258, 524 / 477   40 295 / 371, 609 / 537   79 379 / 634, 1025 / 941
//   n = 4    8 159 / 172, 284 / 231   16 190 / 233, 378 / 318   26 226 / 337, 517 / 450   53 280 / 569, 823 / 737
//   n = 8    8 339 / 362, 462 / 469   12 365 / 483, 597 / 635   26 439 / 918, 971 / 1172
// The lines lie where white noise gains more than walks lose (n = 2, 4), and where it begins to gain by a fifth (n = 8); n = 1
// could start lower.
bool body_suits(const BodyPlan &p, int n)
{
    if (p.form == BodyForm::TILE) return true;
    const bool tuned = (n & (n - 1)) == 0;
    if (p.form == BodyForm::LANE) return !tuned || p.share >= (n == 1 ? 30.0f : n == 2 ? 26.0f : n == 4 ? 18.0f : 10.0f);
    // (n = 1, B = 8, T = 3e3 80 / 92, T = 1e4 96 / 99; n = 2, T = 6e3 114 / 140, T = 1.5e4 142 / 152: above, what a failed try costs
    // on slowly varying inputs, 20 to 30 us, outweighs it)
    if (p.NC > 0 && n <= 2 && (long long)p.max_ctas * p.NC * p.L > (n == 1 ? 20000 : 64000)) return false;
    if (p.NC > 0) return p.whole_loop || (n > 8 && p.waves <= 2.0f) || (!tuned && n > 8 && p.waves <= (n <= 16 ? 4.0f : n <= 32 ? 5.0f : 6.0f));
    if (!tuned) return true;
    return p.waves >= 0.5f;
}

int launch_tile_units(const BodyArgs &a, float *xs, cudaStream_t st)
{
    const size_t count = (size_t)a.B * a.T * a.m;
    const unsigned blocks = (unsigned)std::min<size_t>((count + 1023) / 1024, 8 * (size_t)sm_count());
    DEER_KERNEL("tile_units_kernel", st, pick(a.n, true).tile_units<<<blocks, 256, 0, st>>>(a.x, xs, count, a.m, a.h0.W_h, a.h0.W_i));
    return DEER_OK;
}

int launch_newton_body(const BodyArgs &a, const BodyPlan &p, cudaStream_t st)
{
    const bool aligned = ((((uintptr_t)a.buf[0] | (uintptr_t)a.buf[1] | (uintptr_t)a.y0 | (uintptr_t)a.u) & 7) == 0);
    const bool v2 = (a.n & 1) == 0 && aligned;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.max_ctas, (unsigned)a.H);
    cfg.blockDim = dim3(32u * (unsigned)p.warps);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    if (p.whole_loop) {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    } else {
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
    }
    cfg.attrs = attr; cfg.numAttrs = 1;
    const BodyKernels k = pick(a.n, v2);
    if (p.form == BodyForm::TILE) {
        occupancy_of((const void *)k.tile(a.m), 32 * p.warps, p.smem);
        DEER_KERNEL("newton_tile_kernel", st, k.tile(a.m)<<<(unsigned)p.max_ctas, 32 * p.warps, p.smem, st>>>(a));
        return DEER_OK;
    }
    if (p.form == BodyForm::LANE) {
        const LaneKernel lk = lane_kernel(a.n, a.m, a.u != nullptr);
        occupancy_of((const void *)lk.kern, 128, p.smem);
        DEER_KERNEL("newton_lane_kernel", st, cudaLaunchKernelEx(&cfg, lk.kern, a));
        return DEER_OK;
    }
    occupancy_of(p.NC > 0 ? (const void *)k.seg : (const void *)k.one, 32 * p.warps, p.smem);      // (the shared-memory opt-in on first use)
    if (p.NC > 0) {
        DEER_KERNEL("newton_segment_kernel", st, cudaLaunchKernelEx(&cfg, k.seg, a, p.NC, p.whole_loop ? 1 : 0));
    } else {
        DEER_KERNEL("newton_body_kernel", st, cudaLaunchKernelEx(&cfg, k.one, a));
    }
    return DEER_OK;
}

}  // namespace deer
