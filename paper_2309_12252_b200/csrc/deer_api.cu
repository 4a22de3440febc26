// C-ABI entry points of the DEER-GRU library: validation, workspace carving,
// kernel sequencing and the Newton loop control.
#include <math.h>
#include <stdio.h>
#include <string.h>
#include <stdlib.h>

#include <algorithm>
#include <chrono>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "common.cuh"
#include "kernels_generic.cuh"
#include "scan_onepass.cuh"
#include "scan_hold4.cuh"
#include "scan_warp8.cuh"
#include "scan_warpn.cuh"
#include "scan_warpn_fused.cuh"
#include "scan_fused_fwd.cuh"
#include "scan_cta64.cuh"
#include "scan_verified.cuh"
#include "scan_umma64.cuh"
#include "scan_fused_fwd64.cuh"
#include "cell_wide.cuh"
#include "vjp_wide.cuh"
#include "newton_body.h"
#include "grad_tile.h"
#include "tile_gemm.h"
#include "multihead.cuh"

namespace deer {

std::atomic<long long> g_launches{0};
static thread_local char t_err[256] = "";

void set_error(cudaError_t e, const char *where)
{
    snprintf(t_err, sizeof(t_err), "%s: %s", where, cudaGetErrorString(e));
}

// ---- per-kernel profiling (off by default; benchmarks switch it on for a separate pass)
struct ProfRec { const char *name; cudaEvent_t e0, e1; };
static std::mutex g_prof_mu;
static std::atomic<bool> g_prof_on{false};
static std::vector<ProfRec> g_prof;

KernelScope::KernelScope(const char *name_, cudaStream_t st_) : name(name_), st(st_)
{
    if (!g_prof_on.load(std::memory_order_relaxed)) return;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) { e0 = e1 = nullptr; return; }
    cudaEventRecord(e0, st);
}

KernelScope::~KernelScope()
{
    if (!e0) return;
    cudaEventRecord(e1, st);
    std::lock_guard<std::mutex> lk(g_prof_mu);
    g_prof.push_back({name, e0, e1});
}

// Bump allocator over the caller's workspace; with base == nullptr it only measures.
struct Carver {
    char *base;
    size_t off = 0;
    explicit Carver(void *b) : base((char *)b) {}
    template <typename T> T *take(size_t count)
    {
        size_t o = off;
        off = align_up(off + count * sizeof(T));
        return base ? (T *)(base + o) : nullptr;
    }
};

static int gen_chunk_len(int T)
{
    int L = (int)ceil(sqrt((double)T));
    if (L < 16) L = 16;
    if (L > 256) L = 256;
    return L;
}

struct ScanWs {
    float *carA, *carB, *starts;
    int L, nch;
    OnePassWs op;        // single-pass path (n in {1,2,4,8}); op.nch == 0 when not applicable
    float *vedge;        // chains with a verified burn-in (scan_verified.cuh)
    unsigned *vflag;
    size_t vchains;
    size_t bytes_without;    // workspace up to here: what a scan needs when it goes without them
};

constexpr int VSCAN_L_MIN = 64, VSCAN_BURN = 64, VSCAN_WARPS = 12;
static_assert(VSCAN_BURN % 16 == 0 && VSCAN_WINDOW <= VSCAN_BURN && VSCAN_BURN <= VSCAN_L_MIN, "every chain but the first has a whole window before it");

static int num_sms();

static bool onepass_ll_aggs(int n) { return n <= 4; }

static int onepass_tile_len(int n, int B, int T, int *sw)
{
    *sw = 0;
    switch (n) {
    case 1: return OnePass<1>::L;
    case 2: return OnePass<2>::L;
    case 4: return OnePass<4>::L;
    case 8: *sw = Warp8::chain_len(B, T, 4 * num_sms()); return Warp8::WARPS * *sw;
    case 16: *sw = WarpN<16>::chain_len(B, T, WarpN<16>::CTAS_PER_SM * num_sms()); return WarpN<16>::WARPS * *sw;
    case 32: *sw = WarpN<32>::chain_len(B, T, WarpN<32>::CTAS_PER_SM * num_sms()); return WarpN<32>::WARPS * *sw;
    case 64: return Cta64::L;
    default: return 0;
    }
}

// Sizes for which chains with a verified burn-in pay: enough matrices that reading them is what the scan takes; its 128 steps
// and the launches behind it that return at once take some 30 us (n = 32: 60).  The chunked scan's time goes with the length of
// a sequence.  (B200, us here / there: n = 4, B = 8, T = 4e4 32 / 25, T = 1e5 42 / 42, B = 1, T = 5e5 34 / 108; n = 8, B = 8,
// T = 5e3 26 / 23, T = 2e4 36 / 38, T = 4e4 43 / 58; n = 16, B = 8, T = 5e3 44 / 41, T = 1e4 51 / 58; n = 32, B = 8, T = 2e3
// 67 / 58, T = 3e3 71 / 76, B = 1, T = 4e3 41 / 49; n = 64, B = 1, T = 1e3 86 / 208.)  n <= 2: the one-thread-per-chain scan
// already runs at 0.7 of the copy rate.
static bool vscan_takes(int n, int B, int T)
{
    const double from = n == 64 || B <= 2 ? 8e6 : n == 32 ? 80e6 : 45e6;      // bytes of J
    return (n == 4 || n == 8 || n == 16 || n == 32 || n == 64) && T >= 3 * VSCAN_L_MIN && (double)B * T * n * n * 4 >= from;
}

static ScanWs carve_scan(Carver &cv, int B, int T, int n)
{
    ScanWs w;
    w.L = gen_chunk_len(T);
    w.nch = (T + w.L - 1) / w.L;
    w.carA = cv.take<float>((size_t)B * w.nch * n * n);
    w.carB = cv.take<float>((size_t)B * w.nch * n);
    w.starts = cv.take<float>((size_t)B * w.nch * n);
    w.op = OnePassWs{};
    int L1 = onepass_tile_len(n, B, T, &w.op.sw);
    if (L1) {
        w.op.nch = (T + L1 - 1) / L1;
        size_t tiles = (size_t)B * w.op.nch;
        w.op.flags = cv.take<unsigned>(tiles);
        // (n <= 4 publish their aggregates as 64-bit {value, flag} words)
        w.op.aggs = cv.take<float>(tiles * (n * n + n) * (onepass_ll_aggs(n) ? 2 : 1));
        w.op.starts = cv.take<unsigned long long>(tiles * n);
        w.op.pfx = nullptr;
        if (n == 16) w.op.pfx = cv.take<float>(tiles * (FusedFwd<16>::WARPS - 1) * FusedFwd<16>::AGG);
        if (n == 32) w.op.pfx = cv.take<float>(tiles * (FusedFwd<32>::WARPS - 1) * FusedFwd<32>::AGG);
    }
    w.bytes_without = cv.off;
    w.vchains = vscan_takes(n, B, T) ? (size_t)B * ((T + VSCAN_L_MIN - 1) / VSCAN_L_MIN) : 0;
    w.vedge = cv.take<float>(w.vchains * 3 * n);
    w.vflag = cv.take<unsigned>(w.vchains);
    return w;
}

constexpr int MAX_DEVICES = 64;
static int g_num_sms[MAX_DEVICES] = {0};
static int num_sms()
{
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= MAX_DEVICES) dev = 0;
    if (!g_num_sms[dev]) {
        int v = 0;
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        g_num_sms[dev] = v > 0 ? v : 148;
    }
    return g_num_sms[dev];
}

// Clears the single-pass scan's flag / state words and counters (needed once per workspace: the
// scans leave them cleared).
static int scan_prep(const ScanArgs &a, const OnePassWs &w, cudaStream_t st)
{
    const size_t tiles = (size_t)a.B * w.nch;
    const size_t agg_words = onepass_ll_aggs(a.n) ? tiles * (size_t)(a.n * a.n + a.n) : 0;
    const size_t words = tiles * (size_t)(a.n + 1) + agg_words;
    unsigned pb = (unsigned)((words + 255) / 256);
    if (pb > 592u) pb = 592u;
    if (pb < 1u) pb = 1u;
    DEER_KERNEL("scan_prep_kernel", st, scan_prep_kernel<<<pb, 256, 0, st>>>(a.st, w.flags, tiles, w.starts, tiles * (size_t)a.n,
                                                      (unsigned long long *)w.aggs, agg_words));
    return DEER_OK;
}

// Resolver warps per resolver CTA x sequences one warp can serve, for the kernel that scans size n.
static int resolver_cta_capacity(int n, bool umma)
{
    switch (n) {
    case 1: return OnePass<1>::WARPS * OnePass<1>::MAX_SEQ_PER_WARP;
    case 2: return OnePass<2>::WARPS * OnePass<2>::MAX_SEQ_PER_WARP;
    case 4: return OnePass<4>::WARPS * OnePass<4>::MAX_SEQ_PER_WARP;
    case 8: return Warp8::RES_WARPS * OnePass<8>::MAX_SEQ_PER_WARP;
    case 16: return WarpN<16>::RES_WARPS * WarpN<16>::MAX_SEQ_PER_WARP;
    case 32: return WarpN<32>::RES_WARPS * WarpN<32>::MAX_SEQ_PER_WARP;
    case 64: return umma ? Umma64::RES_WARPS * Umma64::MAX_SEQ_PER_WARP : Cta64::RES_WARPS * Cta64::MAX_SEQ_PER_WARP;
    default: return 0;
    }
}

// Resolver CTAs of a single-pass launch: one warp per sequence up to res_cap CTAs, then several
// sequences per warp, and as many CTAs as the batch needs at max_seq_per_warp sequences per warp.
static int resolver_ctas(int B, int res_warps, int max_seq_per_warp, int res_cap)
{
    int R = (B + res_warps - 1) / res_warps;
    if (R > res_cap) R = res_cap;
    const int per_cta_cap = res_warps * max_seq_per_warp;
    const int need = (B + per_cta_cap - 1) / per_cta_cap;
    return need > R ? need : R;
}

// Resolver CTAs only spin; the workers that feed them must be resident beside them.  At least one CTA
// per SM is resident whatever the kernel, so the single-pass path is taken only while the resolvers a
// batch needs fit a quarter of the SMs; larger batches use the three-level scan.
static long long single_pass_max_batch(int n, bool umma)
{
    return (long long)(num_sms() / 4) * resolver_cta_capacity(n, umma);
}

// n = 16, 32: warps of a resolver CTA that resolve.  A resolver CTA's staging area is shared by its resolving warps,
// and the walk over ONE sequence's tiles is the serial part of a scan: small batches give each sequence a deeper ring.
static int big_res_warps(int B) { return B <= 4 ? 1 : B <= 8 ? 2 : 4; }
// n = 64 (two resolving warps per CTA at most): one warp with all the CTA's tile slots for small batches
static int res_warps64(int B) { return B <= 8 ? 1 : 2; }

struct PassCfg {
    const char *name;
    int threads;
    size_t smem;
    int res_warps;          // resolver warps per resolver CTA
    int max_seq_per_warp;
    int cta_cap;            // CTAs per SM at most
    int res_cap;            // resolver CTAs before warps take several sequences
};

// One persistent launch: grid = resident CTAs (or fewer when there are few tiles); the first
// `resolvers` role tickets become resolver CTAs.
template <typename Kern>
static int launch_single_pass(Kern kern, int (&occ_dev)[MAX_DEVICES], const PassCfg &c, ScanArgs a, OnePassWs w, bool prep,
                              cudaStream_t st)
{
    // the shared-memory opt-in and the occupancy are per device: looked up on each device's first launch
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= MAX_DEVICES) dev = 0;
    int &occ = occ_dev[dev];
    if (!occ) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)c.smem);
        if (e != cudaSuccess) { set_error(e, "cudaFuncSetAttribute(single-pass scan)"); return DEER_ERR_CUDA; }
        int o = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, c.threads, c.smem);
        if (e != cudaSuccess || o < 1) { set_error(e, "occupancy(single-pass scan)"); return DEER_ERR_CUDA; }
        occ = o < c.cta_cap ? o : c.cta_cap;
    }
    const size_t tiles = (size_t)a.B * w.nch;
    const size_t resident = (size_t)num_sms() * occ;
    const int R = resolver_ctas(a.B, c.res_warps, c.max_seq_per_warp, c.res_cap);
    if ((size_t)R * 4 > resident) {      // (scan_is_single_pass keeps such batches off this path)
        snprintf(t_err, sizeof(t_err), "single-pass scan: %d resolver CTAs for %zu resident", R, resident);
        return DEER_ERR_INVALID_ARG;
    }
    w.resolvers = R;
    const size_t want = tiles + (size_t)R;
    unsigned grid = (unsigned)(want < resident ? want : resident);
    if (grid < (unsigned)R + 1u) grid = (unsigned)R + 1u;
    int Wd = 8;
    if (Wd > w.nch) Wd = w.nch;
    w.Wd = Wd;
    w.nwin = (w.nch + Wd - 1) / Wd;
    w.total_ids = (unsigned)((size_t)w.nwin * a.B * Wd);
    int rc;
    if (prep && (rc = scan_prep(a, w, st)) != DEER_OK) return rc;
    DEER_KERNEL_PDL(c.name, a.n <= 8, st, kern, grid, (unsigned)c.threads, c.smem, a, w);
    return DEER_OK;
}

template <int N, bool REV>
static int launch_onepass(ScanArgs a, OnePassWs w, bool prep, cudaStream_t st)
{
    using C = OnePass<N>;
    static int occ[MAX_DEVICES] = {0};
    const PassCfg c{"scan_onepass_kernel", C::THREADS, C::SMEM, C::WARPS, C::MAX_SEQ_PER_WARP, 32, 8};
    return launch_single_pass(scan_onepass_kernel<N, REV>, occ, c, a, w, prep, st);
}

template <bool REV>
static int launch_hold4(ScanArgs a, OnePassWs w, bool prep, cudaStream_t st)
{
    using C = OnePass<4>;
    static int occ[MAX_DEVICES] = {0};
    const PassCfg c{"scan_hold4_kernel", C::THREADS, Hold4::SMEM, C::WARPS, C::MAX_SEQ_PER_WARP, 32, 8};
    return launch_single_pass(scan_hold4_kernel<REV>, occ, c, a, w, prep, st);
}

template <bool REV>
static int launch_warp8(ScanArgs a, OnePassWs w, bool prep, cudaStream_t st)
{
    using C = Warp8;
    static int occ[MAX_DEVICES] = {0};
    const PassCfg c{"scan_warp8_kernel", C::THREADS, C::SMEM, C::RES_WARPS, OnePass<8>::MAX_SEQ_PER_WARP, 4, 8};
    return launch_single_pass(scan_warp8_kernel<REV>, occ, c, a, w, prep, st);
}

template <int N, bool REV>
static int launch_warpn(ScanArgs a, OnePassWs w, bool prep, cudaStream_t st)
{
    using C = WarpN<N>;
    static int occ[MAX_DEVICES] = {0};
    w.res_warps = big_res_warps(a.B);
    const PassCfg c{"scan_warpn_kernel", C::THREADS, C::SMEM, w.res_warps, C::MAX_SEQ_PER_WARP, 8, 8};
    return launch_single_pass(scan_warpn_kernel<N, REV>, occ, c, a, w, prep, st);
}

// scans that generate J_t from coefficient rows (a.J) and a.Wh
template <int N, bool REV>
static int launch_warpnf(ScanArgs a, OnePassWs w, bool prep, cudaStream_t st)
{
    using C = WarpNF<N, REV>;
    static int occ[MAX_DEVICES] = {0};
    w.res_warps = big_res_warps(a.B);
    const PassCfg c{"scan_warpnf_kernel", C::THREADS, C::SMEM, w.res_warps, C::MAX_SEQ_PER_WARP, 8, 8};
    return launch_single_pass(scan_warpnf_kernel<N, REV>, occ, c, a, w, prep, st);
}

// forward scan of deer_gru_eval in the Newton-update form, two launches: chunk reduce + carries, then the
// replay of all chains (16 per warp in lockstep)
template <int N>
static int launch_fused_fwd(ScanArgs a, OnePassWs w, bool prep, cudaStream_t st)
{
    using C = FusedFwd<N>;
    static int occ[MAX_DEVICES] = {0};
    static int occ_apply[MAX_DEVICES] = {0};
    w.res_warps = big_res_warps(a.B);
    const PassCfg c{"scan_fused_reduce_kernel", C::THREADS, C::SMEM, w.res_warps, C::MAX_SEQ_PER_WARP, 8, 8};
    int rc = launch_single_pass(scan_fused_reduce_kernel<N>, occ, c, a, w, prep, st);
    if (rc != DEER_OK) return rc;
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= MAX_DEVICES) dev = 0;
    if (!occ_apply[dev]) {
        cudaError_t e = cudaFuncSetAttribute(scan_fused_apply_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::A_SMEM);
        if (e != cudaSuccess) { set_error(e, "cudaFuncSetAttribute(scan apply)"); return DEER_ERR_CUDA; }
        int o = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, scan_fused_apply_kernel<N>, C::A_THREADS, C::A_SMEM);
        if (e != cudaSuccess || o < 1) { set_error(e, "occupancy(scan apply)"); return DEER_ERR_CUDA; }
        occ_apply[dev] = o;
    }
    const long long nchain = (a.T + w.sw - 1) / w.sw;
    const long long groups = ((long long)a.B * nchain + C::ROWS - 1) / C::ROWS;
    const long long want = (groups + C::A_WARPS - 1) / C::A_WARPS;
    const long long resident = (long long)num_sms() * occ_apply[dev];
    const unsigned grid = (unsigned)(want < resident ? want : resident);
    DEER_KERNEL_PDL("scan_fused_apply_kernel", false, st, scan_fused_apply_kernel<N>, grid, (unsigned)C::A_THREADS, C::A_SMEM, a, w);
    return DEER_OK;
}

// n = 64: the same two launches (a CTA of four warps per chain; the replay kernel reads W_h^T from shared memory)
static int launch_fused_fwd64(ScanArgs a, OnePassWs w, bool prep, cudaStream_t st)
{
    using C = FusedFwd<64>;
    static int occ[MAX_DEVICES] = {0};
    static int occ_apply[MAX_DEVICES] = {0};
    w.sw = C::L;                               // a tile is one chain
    w.res_warps = res_warps64(a.B);
    const PassCfg c{"scan_fused_reduce64_kernel", C::THREADS, C::SMEM, w.res_warps, C::MAX_SEQ_PER_WARP, 4, 16};
    int rc = launch_single_pass(scan_fused_reduce64_kernel, occ, c, a, w, prep, st);
    if (rc != DEER_OK) return rc;
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= MAX_DEVICES) dev = 0;
    if (!occ_apply[dev]) {
        cudaError_t e = cudaFuncSetAttribute(scan_fused_apply64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::P_SMEM);
        if (e != cudaSuccess) { set_error(e, "cudaFuncSetAttribute(scan apply)"); return DEER_ERR_CUDA; }
        int o = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, scan_fused_apply64_kernel, C::P_THREADS, C::P_SMEM);
        if (e != cudaSuccess || o < 1) { set_error(e, "occupancy(scan apply)"); return DEER_ERR_CUDA; }
        occ_apply[dev] = o;
    }
    const long long nchain = (a.T + w.sw - 1) / w.sw;
    const long long groups = ((long long)a.B * nchain + C::ROWS - 1) / C::ROWS;
    const long long want = (groups + C::P_PAIRS - 1) / C::P_PAIRS;
    const long long resident = (long long)num_sms() * occ_apply[dev];
    const unsigned grid = (unsigned)(want < resident ? want : resident);
    DEER_KERNEL_PDL("scan_fused_apply_kernel", false, st, scan_fused_apply64_kernel, grid, (unsigned)C::P_THREADS, C::P_SMEM, a, w);
    return DEER_OK;
}

template <bool REV>
static int launch_cta64(ScanArgs a, OnePassWs w, bool prep, cudaStream_t st)
{
    using C = Cta64;
    static int occ[MAX_DEVICES] = {0};
    w.res_warps = res_warps64(a.B);
    const PassCfg c{"scan_cta64_kernel", C::THREADS, C::SMEM, w.res_warps, C::MAX_SEQ_PER_WARP, 8, 16};
    return launch_single_pass(scan_cta64_kernel<REV>, occ, c, a, w, prep, st);
}

template <bool REV>
static int launch_umma64(ScanArgs a, OnePassWs w, bool prep, cudaStream_t st)
{
    using C = Umma64;
    static int occ[MAX_DEVICES] = {0};
    w.res_warps = C::RES_WARPS;
    const PassCfg c{"scan_umma64_kernel", C::THREADS, C::SMEM, C::RES_WARPS, C::MAX_SEQ_PER_WARP, 2, 8};
    return launch_single_pass(scan_umma64_kernel<REV>, occ, c, a, w, prep, st);
}

static int scan_onepass(ScanArgs a, OnePassWs w, bool prep, int flags, cudaStream_t st)
{
    const bool umma = (flags & DEER_FLAG_TCGEN05) != 0;
    switch (a.n * 2 + (a.reverse ? 1 : 0)) {
    case 2: return launch_onepass<1, false>(a, w, prep, st);
    case 3: return launch_onepass<1, true>(a, w, prep, st);
    case 4: return launch_onepass<2, false>(a, w, prep, st);
    case 5: return launch_onepass<2, true>(a, w, prep, st);
    case 8: return launch_hold4<false>(a, w, prep, st);
    case 9: return launch_hold4<true>(a, w, prep, st);
    case 16: return launch_warp8<false>(a, w, prep, st);
    case 17: return launch_warp8<true>(a, w, prep, st);
    case 32: return a.Wh ? (a.residual ? launch_fused_fwd<16>(a, w, prep, st) : launch_warpnf<16, false>(a, w, prep, st))
                         : launch_warpn<16, false>(a, w, prep, st);
    case 33: return a.Wh ? launch_warpnf<16, true>(a, w, prep, st) : launch_warpn<16, true>(a, w, prep, st);
    case 64: return a.Wh ? (a.residual ? launch_fused_fwd<32>(a, w, prep, st) : launch_warpnf<32, false>(a, w, prep, st))
                         : launch_warpn<32, false>(a, w, prep, st);
    case 65: return a.Wh ? launch_warpnf<32, true>(a, w, prep, st) : launch_warpn<32, true>(a, w, prep, st);
    case 128: return umma ? launch_umma64<false>(a, w, prep, st)
                          : (a.Wh && a.residual) ? launch_fused_fwd64(a, w, prep, st) : launch_cta64<false>(a, w, prep, st);
    case 129: return umma ? launch_umma64<true>(a, w, prep, st) : launch_cta64<true>(a, w, prep, st);
    default: return DEER_ERR_UNSUPPORTED_N;
    }
}

// The limit belongs to the function on the device and not to a launch: it only ever grows, or a call in one thread would lower it
// between another's opt-in and launch.
static int opt_in_smem(const void *fn, size_t bytes)
{
    if (bytes <= 48 * 1024) return DEER_OK;
    static std::mutex mu;
    static std::map<std::pair<const void *, int>, size_t> most;
    int dev = 0;
    DEER_CHECK_CUDA(cudaGetDevice(&dev), "cudaGetDevice");
    std::lock_guard<std::mutex> lk(mu);
    size_t &m = most[{fn, dev}];
    DEER_CHECK_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)std::max(m, bytes)), "cudaFuncSetAttribute");
    m = std::max(m, bytes);
    return DEER_OK;
}

// Three-level scan with the generic kernels.
static int scan_generic(ScanArgs a, cudaStream_t st)
{
    const int n = a.n, nn = n * n;
    size_t sm_red = sizeof(float) * (3 * nn + 2 * n);
    size_t sm_car = sizeof(float) * (nn + n);
    int rc;
    if ((rc = opt_in_smem((const void *)gen_reduce_kernel, sm_red)) != DEER_OK) return rc;
    dim3 grid(a.nch, a.B);
    if (a.nch > 1) {
        DEER_KERNEL("gen_reduce_kernel", st, gen_reduce_kernel<<<grid, GEN_THREADS, sm_red, st>>>(a));
    }
    DEER_KERNEL("gen_carry_kernel", st, gen_carry_kernel<<<a.B, GEN_THREADS, sm_car, st>>>(a));
    DEER_KERNEL("gen_apply_kernel", st, gen_apply_kernel<<<grid, GEN_THREADS, sm_car, st>>>(a));
    return DEER_OK;
}

static bool scan_is_single_pass(const ScanArgs &a, const ScanWs &w, int flags)
{
    const bool aligned = (((uintptr_t)a.J | (uintptr_t)a.b | (uintptr_t)a.y) & 15) == 0;
    return !(flags & DEER_FLAG_GENERIC) && w.op.nch > 0 && aligned &&
           a.B <= single_pass_max_batch(a.n, (flags & DEER_FLAG_TCGEN05) != 0);
}

// prep: clear the single-pass scan's words first (false when the previous scan on this workspace
// left them cleared)
static void apply_test_flags(ScanArgs &a, int flags)
{
    if (flags & DEER_FLAG_EXPIRE_WAITS) { a.spin_limit = 4u; a.no_resolve = 1; }
}

template <int N>
static int launch_vscan_n(const VScanArgs &v, bool rev, long long chains, cudaStream_t st)
{
    using C = VScan<N>;
    const unsigned grid = (unsigned)((chains + C::WARPS * C::CPW - 1) / (C::WARPS * C::CPW));
    if (rev) { DEER_KERNEL("scan_verified_kernel", st, scan_verified_kernel<N, true><<<grid, 128, 0, st>>>(v)); }
    else { DEER_KERNEL("scan_verified_kernel", st, scan_verified_kernel<N, false><<<grid, 128, 0, st>>>(v)); }
    return DEER_OK;
}

// Stand-alone solves: chains with a verified burn-in first; the kernels behind it return at once when it succeeded.
static int launch_vscan(const ScanArgs &a, const ScanWs &w, cudaStream_t st)
{
    VScanArgs v{a.J, a.b, a.y0, a.y, a.B, a.T, 0, VSCAN_BURN, 1e-6f, a.st, w.vedge, w.vflag};
    // chains: VSCAN_WARPS per SM (what keeps enough bytes in flight), fewer positions each only down to VSCAN_L_MIN
    const int warps = VSCAN_WARPS, per_warp = a.n < 32 ? 32 / a.n : 1;
    const long long target = (long long)num_sms() * warps * per_warp;
    long long L = ((long long)a.B * a.T + target - 1) / target;
    v.L = (int)std::min<long long>(std::max<long long>(L, VSCAN_L_MIN), a.T);
    const long long chains = (long long)a.B * ((a.T + v.L - 1) / v.L);
    DEER_CHECK_CUDA(cudaMemsetAsync(w.vflag, 0, sizeof(unsigned) * (size_t)chains, st), "clear boundary flags");
    switch (a.n) {
    case 4: return launch_vscan_n<4>(v, a.reverse != 0, chains, st);
    case 8: return launch_vscan_n<8>(v, a.reverse != 0, chains, st);
    case 16: return launch_vscan_n<16>(v, a.reverse != 0, chains, st);
    case 32: return launch_vscan_n<32>(v, a.reverse != 0, chains, st);
    default: return launch_vscan_n<64>(v, a.reverse != 0, chains, st);
    }
}

// verified: the caller leaves a.st->done to this scan (a stand-alone solve, no loop control)
static int run_scan(ScanArgs a, const ScanWs &w, int flags, cudaStream_t st, bool prep = true, bool verified = false)
{
    apply_test_flags(a, flags);
    if (verified && w.vchains > 0 && !a.Wh && !(flags & (DEER_FLAG_GENERIC | DEER_FLAG_TCGEN05 | DEER_FLAG_EXPIRE_WAITS)) &&
        ((((uintptr_t)a.J) & 15) == 0)) {
        int rc = launch_vscan(a, w, st);
        if (rc != DEER_OK) return rc;
    }
    if (scan_is_single_pass(a, w, flags)) return scan_onepass(a, w.op, prep, flags, st);
    return scan_generic(a, st);
}

// tensor-core affine map (K = inputs, nout = outputs; see affine_mma_kernel)
template <int NB_MAX, bool WT>
static int launch_affine_mma(const float *in, const float *W, const float *bias, float *out, size_t N, int K, int nout,
                             cudaStream_t st, const StatusBlock *unless)
{
    const size_t sm = sizeof(float) * 2 * (size_t)K * (nout + 4);
    int rc;
    if ((rc = opt_in_smem((const void *)affine_mma_kernel<NB_MAX, WT>, sm)) != DEER_OK) return rc;
    const size_t tiles = (N + 127) / 128;
    const size_t per_sm = sm > 110 * 1024 ? 1 : 2;
    const size_t cap = (size_t)num_sms() * per_sm;
    const unsigned blocks = (unsigned)(tiles < cap ? tiles : cap);
    DEER_KERNEL("affine_mma_kernel", st, (affine_mma_kernel<NB_MAX, WT><<<blocks, 256, sm, st>>>(in, W, bias, out, N, K, nout, unless)));
    return DEER_OK;
}

// out[e][g] = bias[g] + sum_k W[g][k] in[e][k]   (wt_given: W is stored [k][g]; bias may be null; unless: nothing to do once
// that block's done is set)
static int run_affine(const float *in, const float *W, const float *bias, float *out, size_t N, int m, int n3,
                      int wt_given, cudaStream_t st, const StatusBlock *unless = nullptr)
{
    // tensor-core path: K and the output count multiples of 8, 8-byte aligned rows, weights fit shared memory
    const bool aligned8 = (((uintptr_t)in | (uintptr_t)out) & 7) == 0;
    if (aligned8 && m % 8 == 0 && m >= 16 && n3 % 8 == 0 && n3 <= 192 &&
        sizeof(float) * 2 * (size_t)m * (n3 + 4) <= 200 * 1024) {
        if (n3 <= 64) return wt_given ? launch_affine_mma<8, true>(in, W, bias, out, N, m, n3, st, unless)
                                      : launch_affine_mma<8, false>(in, W, bias, out, N, m, n3, st, unless);
        if (n3 <= 96) return wt_given ? launch_affine_mma<12, true>(in, W, bias, out, N, m, n3, st, unless)
                                      : launch_affine_mma<12, false>(in, W, bias, out, N, m, n3, st, unless);
        return wt_given ? launch_affine_mma<24, true>(in, W, bias, out, N, m, n3, st, unless)
                        : launch_affine_mma<24, false>(in, W, bias, out, N, m, n3, st, unless);
    }
    int G = 256 / n3;
    while (G > 1 && sizeof(float) * (size_t)G * PROJ_PP * (m + 1) > 64 * 1024) --G;
    const size_t sm = sizeof(float) * ((size_t)m * n3 + (size_t)G * PROJ_PP * (m + 1));
    if (G < 1 || sm > 200 * 1024) return DEER_ERR_UNSUPPORTED_N;
    int rc;
    if ((rc = opt_in_smem((const void *)proj_tiled_kernel, sm)) != DEER_OK) return rc;
    const size_t tiles = (N + (size_t)G * PROJ_PP - 1) / ((size_t)G * PROJ_PP);
    const size_t cap = (size_t)num_sms() * 8;
    const unsigned blocks = (unsigned)(tiles < cap ? tiles : cap);
    const int threads = (n3 * G + 31) / 32 * 32;
    DEER_KERNEL("proj_tiled_kernel", st,
                proj_tiled_kernel<<<blocks, threads, sm, st>>>(in, W, bias, out, N, m, n3, G, wt_given, unless));
    return DEER_OK;
}

static int run_proj(const deer_gru_params *p, const float *x, float *u, size_t N, cudaStream_t st, const StatusBlock *unless = nullptr)
{
    const int n3 = 3 * p->n, m = p->m;
    if (n3 <= 256 && sizeof(float) * ((size_t)m * n3 + (size_t)PROJ_PP * (m + 1)) <= 200 * 1024)
        return run_affine(x, p->W_i, p->b_i, u, N, m, n3, 0, st, unless);
    size_t total = N * (size_t)n3;
    unsigned blocks = (unsigned)((total + 255) / 256);
    DEER_KERNEL("proj_kernel", st, proj_kernel<<<blocks, 256, 0, st>>>(x, p->W_i, p->b_i, u, N, m, n3, unless));
    return DEER_OK;
}

template <int N> static int launch_cell_wide(CellArgs c, cudaStream_t st)
{
    using C = CellWide<N>;
    int rc;
    if ((rc = opt_in_smem((const void *)cell_wide_kernel<N>, C::SMEM)) != DEER_OK) return rc;
    const size_t total = (size_t)c.B * c.T;
    const size_t tiles = (total + C::PT - 1) / C::PT;
    const size_t per_sm = (200 * 1024) / C::SMEM;
    const size_t cap = (size_t)num_sms() * (per_sm > 4 ? 4 : per_sm);
    const unsigned blocks = (unsigned)(tiles < cap ? tiles : cap);
    DEER_KERNEL_PDL("cell_wide_kernel", false, st, cell_wide_kernel<N>, blocks, (unsigned)C::THREADS, C::SMEM, c);
    return DEER_OK;
}

// coefficient rows + rhs only (the scan builds J_t): the hidden contraction on tensor cores
// the tensor-core coefficient cell can contract the input projection itself (no u buffer, no projection pass)
static bool coef_cell_projects(int n, int m, const float *x)
{
    return (n == 32 || n == 16) && m % 8 == 0 && m >= 8 && m <= 64 && (((uintptr_t)x) & 7) == 0;
}

template <int N> static int launch_cell_coef_mma(CellArgs c, cudaStream_t st)
{
    const bool proj = c.u == nullptr;
    const size_t SM = sizeof(float) * (2 * (size_t)N * (3 * N + 4) + 6 * N + (proj ? 2 * (size_t)c.m * (3 * N + 4) : 0));
    int rc;
    const size_t total = (size_t)c.B * c.T;
    const size_t tiles = (total + 127) / 128;
    const size_t cap = (size_t)num_sms() * 2;          // (the kernel's launch bounds: two CTAs per SM; one wave, the weights split once per CTA)
    const unsigned blocks = (unsigned)(tiles < cap ? tiles : cap);
    if (proj) {
        if ((rc = opt_in_smem((const void *)cell_coef_mma_kernel<N, true>, SM)) != DEER_OK) return rc;
        DEER_KERNEL_PDL("cell_coef_mma_kernel", false, st, (cell_coef_mma_kernel<N, true>), blocks, 256u, SM, c);
    } else {
        if ((rc = opt_in_smem((const void *)cell_coef_mma_kernel<N, false>, SM)) != DEER_OK) return rc;
        DEER_KERNEL_PDL("cell_coef_mma_kernel", false, st, (cell_coef_mma_kernel<N, false>), blocks, 256u, SM, c);
    }
    return DEER_OK;
}

template <int N> static int launch_cell_small(CellArgs c, cudaStream_t st)
{
    const size_t total = (size_t)c.B * c.T;
    const size_t epb = 256 / N;
    size_t blocks = (total + epb - 1) / epb;
    // three CTAs are resident per SM (registers): a small problem runs as one persistent wave, a large one
    // is split finer so that the last wave is balanced (measured: 21.4 vs 23.5 us on config 2; 6.4 vs 7.9 ms at T = 1e6)
    const size_t resident = (size_t)num_sms() * 3;
    const size_t cap = blocks < 16 * resident ? resident : (size_t)num_sms() * 8;
    if (blocks > cap) blocks = cap;
    const unsigned gb = (unsigned)blocks;
    if (c.u) { DEER_KERNEL_PDL("cell_small_kernel", true, st, (cell_small_kernel<N, 0>), gb, 256u, 0, c); return DEER_OK; }
    switch (c.m) {
    case 1: DEER_KERNEL_PDL("cell_small_kernel", true, st, (cell_small_kernel<N, 1>), gb, 256u, 0, c); break;
    case 2: DEER_KERNEL_PDL("cell_small_kernel", true, st, (cell_small_kernel<N, 2>), gb, 256u, 0, c); break;
    case 4: DEER_KERNEL_PDL("cell_small_kernel", true, st, (cell_small_kernel<N, 4>), gb, 256u, 0, c); break;
    case 8: DEER_KERNEL_PDL("cell_small_kernel", true, st, (cell_small_kernel<N, 8>), gb, 256u, 0, c); break;
    default: return DEER_ERR_INVALID_ARG;
    }
    return DEER_OK;
}

// the cell kernel can project x itself (no u buffer, no proj pass) for these sizes
static bool cell_projects(int n, int m)
{
    return (n == 1 || n == 2 || n == 4 || n == 8) && (m == 1 || m == 2 || m == 4 || m == 8);
}

static int run_cell(CellArgs c, cudaStream_t st, bool generic = false)
{
    const bool aligned = (((uintptr_t)c.y | (uintptr_t)c.y0 | (uintptr_t)c.J) & 15) == 0;
    if (aligned && !generic) {
        switch (c.n) {
        case 1: return launch_cell_small<1>(c, st);
        case 2: return launch_cell_small<2>(c, st);
        case 4: return launch_cell_small<4>(c, st);
        case 8: return launch_cell_small<8>(c, st);
        default: break;
        }
        if ((c.u || (c.coef_only && c.residual && coef_cell_projects(c.n, c.m, c.x))) && (((uintptr_t)c.W_h) & 15) == 0) {
            switch (c.n) {
            case 16: return (c.coef_only && !c.u) ? launch_cell_coef_mma<16>(c, st) : launch_cell_wide<16>(c, st);
            case 32: return c.coef_only ? launch_cell_coef_mma<32>(c, st) : launch_cell_wide<32>(c, st);
            case 64: return (c.coef_only && c.u) ? launch_cell_coef_mma<64>(c, st) : launch_cell_wide<64>(c, st);
            default: break;
            }
        }
    }
    const int n = c.n;
    size_t sm = sizeof(float) * (3 * n * (n + 1) + 3 * n);
    int rc;
    if ((rc = opt_in_smem((const void *)cell_kernel, sm)) != DEER_OK) return rc;
    int threads = 256;
    int epb = threads / n;
    size_t N = (size_t)c.B * c.T;
    unsigned blocks = (unsigned)((N + epb - 1) / epb);
    DEER_KERNEL("cell_kernel", st, cell_kernel<<<blocks, threads, sm, st>>>(c));
    return DEER_OK;
}

template <int N> static int launch_vjp_cell_wide_n(VjpArgs v, cudaStream_t st)
{
    using C = CellWide<N>;
    const size_t sm = sizeof(float) * (3 * N * N + 3 * N + C::PT * C::HS);
    int rc;
    if ((rc = opt_in_smem((const void *)vjp_cell_wide_kernel<N>, sm)) != DEER_OK) return rc;
    const size_t total = (size_t)v.B * v.T;
    const size_t tiles = (total + C::PT - 1) / C::PT;
    const size_t per_sm = (200 * 1024) / sm;
    const size_t cap = (size_t)num_sms() * (per_sm > 4 ? 4 : per_sm);
    const unsigned blocks = (unsigned)(tiles < cap ? tiles : cap);
    DEER_KERNEL("vjp_cell_wide_kernel", st, vjp_cell_wide_kernel<N><<<blocks, C::THREADS, sm, st>>>(v));
    return DEER_OK;
}

static int launch_vjp_cell_wide(VjpArgs v, cudaStream_t st)
{
    switch (v.n) {
    case 16: return launch_vjp_cell_wide_n<16>(v, st);
    case 32: return launch_vjp_cell_wide_n<32>(v, st);
    case 64: return launch_vjp_cell_wide_n<64>(v, st);
    default: return DEER_ERR_UNSUPPORTED_N;
    }
}

static bool valid_sizes(int B, int T, int n, int m)
{
    return B > 0 && T > 0 && n > 0 && m > 0 && (double)B * T * n * n < 9.0e18;
}

static bool supported(int n, int m) { return n >= 1 && n <= 64 && m >= 1 && m <= 1024; }

// ---------------------------------------------------------------- workspace layouts
struct EvalWs {
    StatusBlock *st;
    float *trace;        // [ERR_TRACE_CAP] err after each body (device side of err_trace)
    unsigned long long *diag;   // [B] per-sequence {err bits, inverted index} of the last body
    float *u, *J, *rhs, *yalt;
    float *edge;         // one-launch bodies: states at the boundaries between warps
    unsigned *edge_flag;
    unsigned long long *words;   // whole-loop launches: exchanged maxima (at most one CTA per SM)
    ScanWs scan;
    size_t bytes;
};

// chain groups of a one-launch body at the shortest chain length
static size_t body_groups_max(int B, int T) { return ((size_t)B * ((T + BODY_L_MIN - 1) / BODY_L_MIN) + 15) / 16; }

// ... and of an adjoint launch, idle warps of the last CTA included
static size_t adjoint_groups_max(int B, int T) { return ((size_t)B * ((T + CHAIN_L_MIN - 1) / CHAIN_L_MIN) + 15) / 16 + 8; }

// boundaries of any of a gradient's launches: those of rows_adjoint.cuh lie between warps of 32 / n chains
static size_t adjoint_edges_max(int B, int T, int n)
{
    const size_t chains = (size_t)B * ((T + CHAIN_L_MIN - 1) / CHAIN_L_MIN), unit = n == 4 || n == 8 ? 32 / n : 16;
    return (chains + unit - 1) / unit;
}

static EvalWs carve_eval(void *ws, int B, int T, int n, int m)
{
    (void)m;
    Carver cv(ws);
    EvalWs w;
    size_t N = (size_t)B * T;
    w.st = cv.take<StatusBlock>(1);
    w.trace = cv.take<float>(ERR_TRACE_CAP);
    w.diag = cv.take<unsigned long long>((size_t)B);
    w.u = cv.take<float>(N * 3 * n);
    w.J = cv.take<float>(N * n * n);
    w.rhs = cv.take<float>(N * n);
    w.yalt = cv.take<float>(N * n);
    w.edge = cv.take<float>(body_groups_max(B, T) * 2 * n);
    w.edge_flag = cv.take<unsigned>(body_groups_max(B, T));
    w.words = cv.take<unsigned long long>((size_t)4 * num_sms());
    w.scan = carve_scan(cv, B, T, n);
    w.bytes = cv.off;
    return w;
}

struct ScanOnlyWs {
    StatusBlock *st;
    ScanWs scan;
    size_t bytes;
};

static ScanOnlyWs carve_scan_only(void *ws, int B, int T, int n)
{
    Carver cv(ws);
    ScanOnlyWs w;
    w.st = cv.take<StatusBlock>(1);
    w.scan = carve_scan(cv, B, T, n);
    w.bytes = cv.off;
    return w;
}

constexpr int WGRAD_P = 592;   // slices of the position axis in the parameter-gradient reduction

struct VjpWs {
    StatusBlock *st;
    unsigned *edge_flag;         // directly behind the status block: cleared with it
    float *edge, *starts;
    size_t edges, start_groups;  // boundaries and chain groups that there is room for
    float *u, *J, *rhs, *lam, *dGi, *dGh, *partial, *partial2;
    ScanWs scan;
    size_t bytes;
};

static VjpWs carve_vjp(void *ws, int B, int T, int n, int m)
{
    Carver cv(ws);
    VjpWs w;
    size_t N = (size_t)B * T;
    w.st = cv.take<StatusBlock>(1);
    w.edges = adjoint_edges_max(B, T, n);
    w.edge_flag = cv.take<unsigned>(w.edges);
    w.edge = cv.take<float>(w.edges * ADJ_EDGE(n));
    w.start_groups = adjoint_groups_max(B, T);
    w.starts = cv.take<float>(w.start_groups * adjoint_starts(n));
    w.u = cv.take<float>(N * 3 * n);
    w.J = cv.take<float>(N * n * n);
    w.lam = cv.take<float>(N * n);
    w.dGi = cv.take<float>(N * 3 * n);
    w.dGh = cv.take<float>(N * 3 * n);
    int kmax = (m > n ? m : n) + 1;
    w.partial = cv.take<float>((size_t)WGRAD_P * 3 * n * kmax);
    w.partial2 = cv.take<float>((size_t)WGRAD_P * 3 * n * kmax);
    w.scan = carve_scan(cv, B, T, n);
    w.rhs = nullptr;
    w.bytes = cv.off;
    return w;
}

struct ClsWs {
    float *y1, *y2, *gyA, *gyB, *pool_partial, *pooled, *dlog, *gpool, *loss;
    void *inner;
    size_t inner_bytes, bytes;
};
constexpr int POOL_SEGS = 64;

static ClsWs carve_cls(void *ws, int B, int T, int n, int m, int ncls)
{
    Carver cv(ws);
    ClsWs w;
    size_t N = (size_t)B * T;
    w.y1 = cv.take<float>(N * n);
    w.y2 = cv.take<float>(N * n);
    w.gyA = cv.take<float>(N * n);
    w.gyB = cv.take<float>(N * n);
    w.pool_partial = cv.take<float>((size_t)B * POOL_SEGS * n);
    w.pooled = cv.take<float>((size_t)B * n);
    w.dlog = cv.take<float>((size_t)B * ncls);
    w.gpool = cv.take<float>((size_t)B * n);
    w.loss = cv.take<float>(64);
    int mm = m > n ? m : n;
    size_t e = carve_eval(nullptr, B, T, n, mm).bytes;
    size_t v = carve_vjp(nullptr, B, T, n, mm).bytes;
    w.inner_bytes = e > v ? e : v;
    w.inner = cv.take<char>(w.inner_bytes);
    w.bytes = cv.off;
    return w;
}

struct OdeWs {
    StatusBlock *st;
    float *J, *rhs;
    ScanWs scan;
    size_t bytes;
};

static OdeWs carve_ode(void *ws, int B, int T, int n)
{
    Carver cv(ws);
    OdeWs w;
    w.st = cv.take<StatusBlock>(1);
    w.J = cv.take<float>((size_t)B * T * n * n);
    w.rhs = cv.take<float>((size_t)B * T * n);
    w.scan = carve_scan(cv, B, T, n);
    w.bytes = cv.off;
    return w;
}

struct LstmWs {
    StatusBlock *st;
    float *trace, *u, *J, *rhs, *yalt;
    ScanWs scan;
    size_t bytes;
};

static LstmWs carve_lstm(void *ws, int B, int T, int k)
{
    Carver cv(ws);
    LstmWs w;
    const size_t N = (size_t)B * T;
    const int n = 2 * k;
    w.st = cv.take<StatusBlock>(1);
    w.trace = cv.take<float>(ERR_TRACE_CAP);
    w.u = cv.take<float>(N * 4 * k);
    w.J = cv.take<float>(N * n * n);
    w.rhs = cv.take<float>(N * n);
    w.yalt = cv.take<float>(N * n);
    w.scan = carve_scan(cv, B, T, n);
    w.bytes = cv.off;
    return w;
}

// multi-head unit: dense batches of one stride group at a time + the inner evaluation / gradient workspace
struct MhWs {
    float *xs, *y0s, *ys, *gys, *dxs, *dy0s;
    void *inner;
    size_t inner_bytes, bytes;
    // all heads as one batch
    BodyHead *heads;
    MhGrad *grads;
    StatusBlock *st;         // [H]
    float *Wc, *bc;          // input weights and biases side by side
    float *u, *yalt, *dGi, *dGh, *edge, *starts, *dy0all, *partial;
    unsigned *edge_flag;
    unsigned long long *words;
    size_t groups, start_groups;
};

constexpr int MH_P_IN = 32;  // slices of the positions in the reduction of the stacked input weights
// ... and of a head's hidden weights: about 16 CTAs per SM over all heads
static int mh_p_hidden(int H) { return std::max(8, std::min(128, 2368 / H)); }

static MhWs carve_mh(void *ws, int H, const int *strides, int B, int T, int n, int m)
{
    Carver cv(ws);
    MhWs w;
    size_t maxN = 0, maxB = 0, inner = 0;
    for (int h = 0; h < H; ++h) {
        const int s = strides[h];
        const int Tp = (T + s - 1) / s;
        const size_t Bs = (size_t)B * s;
        maxN = Bs * Tp > maxN ? Bs * Tp : maxN;
        maxB = Bs > maxB ? Bs : maxB;
        const size_t e = carve_eval(nullptr, (int)Bs, Tp, n, m).bytes, v = carve_vjp(nullptr, (int)Bs, Tp, n, m).bytes;
        inner = e > inner ? e : inner;
        inner = v > inner ? v : inner;
    }
    w.xs = cv.take<float>(maxN * m);
    w.y0s = cv.take<float>(maxB * n);
    w.ys = cv.take<float>(maxN * n);
    w.gys = cv.take<float>(maxN * n);
    w.dxs = cv.take<float>(maxN * m);
    w.dy0s = cv.take<float>(maxB * n);
    w.inner_bytes = inner;
    w.inner = cv.take<char>(inner);
    const size_t N = (size_t)B * T, n3 = 3 * (size_t)n;
    size_t agroups = 0, seqs = 0;
    w.groups = 0;
    for (int h = 0; h < H; ++h) {
        const int Bs = B * strides[h], Tp = (T + strides[h] - 1) / strides[h];
        w.groups += body_groups_max(Bs, Tp) + 1;
        agroups += adjoint_groups_max(Bs, Tp);
        seqs += (size_t)Bs;
    }
    w.heads = cv.take<BodyHead>(H);
    w.grads = cv.take<MhGrad>(H);
    w.st = cv.take<StatusBlock>(H);
    w.Wc = cv.take<float>(H * n3 * m);
    w.bc = cv.take<float>(H * n3);
    w.u = cv.take<float>(N * H * n3);
    w.yalt = cv.take<float>(N * H * n);
    w.dGi = cv.take<float>(N * H * n3);
    w.dGh = cv.take<float>(N * H * n3);
    w.edge = cv.take<float>(w.groups * ADJ_EDGE(n));
    w.edge_flag = cv.take<unsigned>(w.groups);
    w.words = cv.take<unsigned long long>((size_t)4 * num_sms());
    w.start_groups = agroups;
    w.starts = cv.take<float>(agroups * adjoint_starts(n));
    w.dy0all = cv.take<float>(seqs * n);
    w.partial = cv.take<float>(std::max((size_t)MH_P_IN * H * n3 * (m + 1), (size_t)mh_p_hidden(H) * H * n3 * (n + 1)));
    w.bytes = cv.off;
    return w;
}

static int check_mh_args(const deer_gru_params *heads, const int *strides, int H, int B, int T)
{
    if (!heads || !strides || H < 1 || B <= 0 || T <= 0) return DEER_ERR_INVALID_ARG;
    for (int h = 0; h < H; ++h) {
        if (!heads[h].W_i || !heads[h].W_h || !heads[h].b_i || !heads[h].b_h) return DEER_ERR_INVALID_ARG;
        if (heads[h].n != heads[0].n || heads[h].m != heads[0].m || heads[h].n <= 0 || heads[h].m <= 0) return DEER_ERR_INVALID_ARG;
        if (strides[h] < 1 || (long long)B * strides[h] > 0x7fffffffLL) return DEER_ERR_INVALID_ARG;
    }
    if (!supported(heads[0].n, heads[0].m)) return DEER_ERR_UNSUPPORTED_N;
    if (!valid_sizes(B, T, heads[0].n, heads[0].m)) return DEER_ERR_INVALID_ARG;
    return DEER_OK;
}

static unsigned mh_blocks(size_t total);

// strided view -> dense batch and back (128-bit moves when the layout allows)
static int mh_pack(const float *src, float *dst, int B, int T, int s, int Tp, int C, int C_src, int off, cudaStream_t st)
{
    const size_t total = (size_t)B * s * Tp * C;
    const bool v4 = C % 4 == 0 && C_src % 4 == 0 && off % 4 == 0 && ((((uintptr_t)src | (uintptr_t)dst) & 15) == 0);
    if (v4) { DEER_KERNEL("mh_pack_kernel", st, mh_pack_kernel<4><<<mh_blocks(total / 4), 256, 0, st>>>(src, dst, B, T, s, Tp, C, C_src, off)); }
    else { DEER_KERNEL("mh_pack_kernel", st, mh_pack_kernel<1><<<mh_blocks(total), 256, 0, st>>>(src, dst, B, T, s, Tp, C, C_src, off)); }
    return DEER_OK;
}

static int mh_unpack(const float *src, float *dst, int B, int T, int s, int Tp, int C, int C_dst, int off, int accumulate,
                     cudaStream_t st)
{
    const size_t total = (size_t)B * s * Tp * C;
    const bool v4 = C % 4 == 0 && C_dst % 4 == 0 && off % 4 == 0 && ((((uintptr_t)src | (uintptr_t)dst) & 15) == 0);
    if (v4) { DEER_KERNEL("mh_unpack_kernel", st, mh_unpack_kernel<4><<<mh_blocks(total / 4), 256, 0, st>>>(src, dst, B, T, s, Tp, C, C_dst, off, accumulate)); }
    else { DEER_KERNEL("mh_unpack_kernel", st, mh_unpack_kernel<1><<<mh_blocks(total), 256, 0, st>>>(src, dst, B, T, s, Tp, C, C_dst, off, accumulate)); }
    return DEER_OK;
}

static unsigned mh_blocks(size_t total)
{
    size_t b = (total + 255) / 256;
    const size_t cap = (size_t)num_sms() * 8;
    if (b > cap) b = cap;
    return (unsigned)(b < 1 ? 1 : b);
}

static int check_ws(void *ws, size_t have, size_t need)
{
    if (!ws || ((uintptr_t)ws & 255) != 0 || have < need) return DEER_ERR_WORKSPACE;
    return DEER_OK;
}

// ---------------------------------------------------------------- implementation bodies
static int linrec_scan_impl(const float *J, const float *b, const float *y0, int B, int T, int n,
                            int reverse, float *y, void *ws, size_t ws_bytes, int flags,
                            cudaStream_t st)
{
    ScanOnlyWs w = carve_scan_only(ws, B, T, n);
    int rc = check_ws(ws, ws_bytes, w.scan.bytes_without);
    if (rc != DEER_OK) return rc;
    if (ws_bytes < w.bytes) w.scan.vchains = 0;
    DEER_CHECK_CUDA(cudaMemsetAsync(w.st, 0, sizeof(StatusBlock), st), "memset status");
    ScanArgs a{};
    a.J = J; a.b = b; a.y0 = y0; a.y = y; a.yold = nullptr;
    a.B = B; a.T = T; a.n = n; a.reverse = reverse ? 1 : 0;
    a.L = w.scan.L; a.nch = w.scan.nch;
    a.carA = w.scan.carA; a.carB = w.scan.carB; a.starts = w.scan.starts;
    a.st = w.st;
    return run_scan(a, w.scan, flags, st, true, true);
}

// A page-locked record for the result of one evaluation, from a fixed set that is made on first use (8 KB per process).
// An evaluation that finds none free, or no page-locked memory, reads its status with a copy instead.
class HostSlot {
    static constexpr int COUNT = 64;
    static HostResult *base()
    {
        static HostResult *b = []() -> HostResult * {
            void *v = nullptr;
            if (cudaHostAlloc(&v, COUNT * sizeof(HostResult), cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) { cudaGetLastError(); return nullptr; }
            return (HostResult *)v;
        }();
        return b;
    }
    static std::atomic<unsigned long long> &taken() { static std::atomic<unsigned long long> t{0}; return t; }
    int idx = -1;

public:
    HostResult *p = nullptr;
    explicit HostSlot(bool want)
    {
        if (!want || !base()) return;
        for (unsigned long long t = taken().load(); ~t != 0ull;) {
            const int i = __builtin_ctzll(~t);
            if (taken().compare_exchange_weak(t, t | (1ull << i))) { idx = i; p = base() + i; return; }
        }
    }
    ~HostSlot() { if (idx >= 0) taken().fetch_and(~(1ull << idx)); }
    HostSlot(const HostSlot &) = delete;
    HostSlot &operator=(const HostSlot &) = delete;
};

// Reads the record until the loop or the form has ended there, which is before the launches enqueued behind it have drained,
// and returns how; 0 after `us` microseconds, or where the stream has come to its end.
static int record_posted(const HostResult *hr, cudaStream_t st, int us)
{
    const volatile int *done = &hr->done;
    const auto from = std::chrono::steady_clock::now();
    for (unsigned k = 1;; ++k) {
        if (const int how = *done) return how;
        if (k % 16 == 0 && std::chrono::steady_clock::now() - from > std::chrono::microseconds(us)) return 0;
        if (k % 4096 == 0 && cudaStreamQuery(st) != cudaErrorNotReady) return *done;         // (an error is sticky: the caller's synchronisation reports it)
    }
}

// ---- evaluations whose bodies are one launch each (newton_body.cuh)
// The flags that ask for a particular form of the scan are served by the kernels that have that form.
static bool body_takes(int n, int m, int flags)
{
    return !(flags & (DEER_FLAG_GENERIC | DEER_FLAG_MATERIALIZE | DEER_FLAG_TCGEN05 | DEER_FLAG_EXPIRE_WAITS)) &&
           (body_supported(n, m, false) || body_supported(n, m, true));
}

// How long the record is read before the host waits for the stream, in microseconds.  The bias check answers some 10 us after
// its launch, without a body; a longer look costs more at the end of an evaluation (a synchronisation that is entered late,
// 0.7 us) than a form that gives up later gains.
constexpr int BIAS_US = 20, RESULT_US = 20000;

// Chains up to this length get the burn-in that each body calls for (body_verdict); with longer ones a try that fails is dearer
// than what a few steps of them give (n = 1, 224 positions: 370 us either way).  Multi-head units do without: one head whose
// try fails holds up the others (17 heads of 8: 815 -> 1226 us).
constexpr int BODY_L_ADAPT = 64;

// Runs the Newton loop until it ends or the forms give up (hs->done is not BODY_DONE, the iterate after hs->iters bodies in
// buf[hs->iters & 1]).
template <typename CopyOut>
static int eval_one_launch(const deer_gru_params *p, const float *x, const float *y0, int B, int T, float tol, int max_iter,
                           const EvalWs &w, float *const (&buf)[2], int flags, cudaStream_t st, StatusBlock *hs, HostResult *hr,
                           bool &u_done, bool to_host, bool &polled, CopyOut copy_out)
{
    const int n = p->n, m = p->m;
    bool need_u = !body_supported(n, m, false);
    const int first = body_first_burn(n, tol);
    int rc, burn = first;
    BodyArgs a{};
    a.h0 = BodyHead{p->W_i, p->W_h, p->b_i, p->b_h, 1, 0};
    a.x = x; a.y0 = y0;
    a.buf[0] = buf[0]; a.buf[1] = buf[1];
    a.B = B; a.T = T; a.n = n; a.m = m; a.H = 1;
    a.eta = body_eta(n, tol);
    a.expire = (flags & DEER_FLAG_EXPIRE_BODY_WAITS) != 0;
    a.polled = to_host;
    a.st = w.st; a.edge = w.edge; a.edge_flag = w.edge_flag; a.words = w.words;
    a.starts = w.J;                                      // (chains x n floats; nothing else is kept there meanwhile)
    const bool aligned32 = (((uintptr_t)buf[0] | (uintptr_t)buf[1]) & 31) == 0 && (((uintptr_t)y0 | (uintptr_t)p->W_h) & 15) == 0;
    bool tiles = false;
    int tried = -1;                                      // the form launched last (the f16 forms have a second try)
    for (const BodyForm form : {BodyForm::TWO_PHASE, BodyForm::TWO_PHASE, BodyForm::TILE, BodyForm::TILE, BodyForm::LANE, BodyForm::ONE_PHASE, BodyForm::ONE_PHASE}) {
        BodyPlan plan{};
        if ((int)form == tried && form != BodyForm::TILE) {
            // What an operand could not hold was most likely an input: projected inputs go to the accumulators, which have fp32's range.
            if (hs->done != BODY_BEYOND) continue;
            need_u = true;
        }
        if (form == BodyForm::TILE && !aligned32) continue;
        if (form == BodyForm::TILE && tiles) {           // again, with the inputs in units of its own (in the place of u)
            if (hs->done != BODY_UNITS) continue;
            if ((rc = launch_tile_units(a, w.u, st)) != DEER_OK) return rc;
            u_done = false;
            a.x = w.u;
            a.units = 1;
        }
        if (form == BodyForm::ONE_PHASE && tiles) break;             // (what the tiles give up is for the kernels that multiply the Jacobians out)
        const bool have_u = form == BodyForm::LANE ? m > 8 : need_u && form != BodyForm::TILE;
        if (!body_plan(&plan, form, B, T, n, m, have_u, nullptr, 1) || !body_suits(plan, n)) continue;
        a.u = have_u ? w.u : nullptr;
        // n = 32, 64: the two-phase kernel only where it is the whole loop in one launch
        if (form == BodyForm::TWO_PHASE && (n == 32 || n == 64) && aligned32 && m <= 64 && !plan.whole_loop) continue;
        tiles = form == BodyForm::TILE;
        tried = (int)form;
        if (burn > plan.burn_cap) { hs->done = BODY_FALL_BACK; continue; }
        a.L = plan.L;
        a.burn_cap = plan.burn_cap;
        a.adapt = plan.L <= BODY_L_ADAPT;
        a.warm = ((flags & DEER_FLAG_WARM_START) || hs->iters > 0) ? 1 : 0;
        StatusBlock init;
        memset(&init, 0, sizeof(init));
        init.max_iter = max_iter;
        init.tol = tol;
        init.trace = w.trace;
        init.burn = burn == first && !a.warm ? body_start_burn(n, tol, a.adapt != 0) : burn;
        init.iters = hs->iters;
        init.host = hr;
        if (hr) { hr->iters = hs->iters; hr->done = 0; }
        EvalBeginArgs e{};
        if (plan.whole_loop) {
            e.starts = (unsigned long long *)w.edge; e.nstarts = (size_t)plan.edges * n;
            e.agg_words = w.words; e.nagg_words = (size_t)4 * plan.max_ctas;
        } else {
            e.flags = w.edge_flag; e.nflags = (size_t)plan.edges;
        }
        if (T > plan.burn_cap) {
            // a cell initialised to remember for long: where its slowest state, by the bias of its update gate, keeps a tenth
            // over the longest burn-in, no try is made
            e.b_i = p->b_i; e.b_h = p->b_h; e.n = n;
            e.slow = powf(0.1f, 1.0f / (float)plan.burn_cap);
        }
        const unsigned blocks = (unsigned)((e.nflags + e.nstarts + 1023) / 1024);
        DEER_KERNEL("eval_begin_kernel", st, eval_begin_kernel<<<blocks < 1u ? 1u : blocks, 256, 0, st>>>(w.st, init, e));
        if (have_u && !u_done) {
            if ((rc = run_proj(p, x, w.u, (size_t)B * T, st)) != DEER_OK) return rc;
            u_done = true;
        }
        for (int group = 4;; group = 2) {
            const int left = max_iter - hs->iters;
            for (int j = 0; j < (plan.whole_loop ? 1 : left < group ? left : group); ++j) {
                if (hr && *(volatile int *)&hr->done) break;             // (the bias alone has told, or the loop is over already)
                if ((rc = launch_newton_body(a, plan, st)) != DEER_OK) return rc;
            }
            if ((rc = copy_out(false)) != DEER_OK) return rc;
            if (hr) {
                // A result for the host starts on its way, and the next form goes ahead, as soon as the record tells.
                const int end = record_posted(hr, st, to_host ? RESULT_US : BIAS_US);
                polled = to_host && end == BODY_DONE;
                if ((end == 0 || end == BODY_DONE || end == BODY_TIMED_OUT) && !polled) DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
                hs->iters = hr->iters; hs->done = hr->done; hs->burn = hr->burn; hs->err_last_bits = hr->err_bits;
                if (hs->done == BODY_TIMED_OUT || (plan.whole_loop && !hs->done)) return DEER_ERR_DEVICE_TIMEOUT;
            } else {
                DEER_CHECK_CUDA(cudaMemcpyAsync(hs, w.st, 48, cudaMemcpyDeviceToHost, st), "read status");
                DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
                if (hs->flags & FLAG_TIMEOUT) return DEER_ERR_DEVICE_TIMEOUT;
            }
            if (hs->done) break;
        }
        if (hs->done == BODY_DONE) return copy_out(true);
        if (hs->done != BODY_BEYOND) burn = hs->burn;
        else if (tiles || have_u) break;                 // (no other form has a wider range)
    }
    return DEER_OK;                                      // (hs->done == BODY_FALL_BACK or BODY_BEYOND)
}

// Results up to this size are copied to host memory before it is known that they are final: the copy is then enqueued while the
// bodies run, and one that proves to be in vain takes 40 us of the link at most.  (n = 8, m = 4, B = 4, us per call, early /
// not: T = 2,000 96 / 97, T = 16,000 (2 MB) 162 / 166, T = 32,000 241 / 240.  What early copies of large results cost: n = m =
// 32, B = 16, T = 1e5, a cell that remembers for up to 1,000 steps 24.3 / 18.2 ms, random walks 16.4 / 10.9 ms.)
constexpr size_t HOST_COPY_EARLY = 2 << 20;

static int eval_status(float e, float tol)
{
    if (!isfinite(e)) return DEER_NONFINITE;
    return e > tol && !(tol < 0.0f) ? DEER_NOT_CONVERGED : DEER_OK;
}

// copy_st / copy_ev (optional): the stream the copy to y_host is enqueued on, and an event to order it behind `st`.
// y_host (optional, host memory): the result is also copied there, after a device-side selection of the buffer that holds the
// current iterate, once the loop has ended.  A small result is copied behind every group of bodies, whether or not it is the
// last: an evaluation that converges within its first group then costs one host synchronisation in all.
static int gru_eval_impl(const deer_gru_params *p, const float *x, const float *y0, int B, int T,
                         float tol, int max_iter, float *y, int *iters, float *err,
                         float *err_trace, void *ws, size_t ws_bytes, int flags, cudaStream_t st,
                         float *y_host = nullptr, float *err_b = nullptr, unsigned long long *err_argmax = nullptr,
                         cudaStream_t copy_st = nullptr, cudaEvent_t copy_ev = nullptr, int bodies_done = 0, int *burn_in = nullptr)
{
    const int n = p->n, m = p->m;
    EvalWs w = carve_eval(ws, B, T, n, m);
    int rc = check_ws(ws, ws_bytes, w.bytes);
    if (rc != DEER_OK) return rc;
    const size_t N = (size_t)B * T;
    float *buf[2] = {y, w.yalt};
    StatusBlock hs;
    memset(&hs, 0, sizeof(hs));
    // ended: the loop has
    const bool copy_early = N * n * sizeof(float) <= HOST_COPY_EARLY;
    bool polled = false;                       // the end of the loop was read from the record
    auto copy_out = [&](bool ended) -> int {
        if (!y_host || ended == copy_early) return DEER_OK;
        if (ended && polled && hs.done == BODY_DONE && (hs.iters & 1) == 0) {
            // the record has told that the result is complete, and it is where it belongs: nothing to wait for (three calls less
            // between the last body and the copy: n = m = 32, B = 16, T = 1e5 6773 -> 6742 us)
            DEER_CHECK_CUDA(cudaMemcpyAsync(y_host, y, N * n * sizeof(float), cudaMemcpyDeviceToHost, copy_st ? copy_st : st), "copy result to host");
            return DEER_OK;
        }
        size_t words = N * n / 4;
        unsigned blocks = (unsigned)((words + 1023) / 1024);
        const unsigned cap = 4u * (unsigned)num_sms();
        if (blocks > cap) blocks = cap;
        if (blocks < 1u) blocks = 1u;
        DEER_KERNEL("result_select_kernel", st, result_select_kernel<<<blocks, 256, 0, st>>>(w.st, y, w.yalt, N * n));
        if (copy_st) {      // the result leaves on a stream of its own, behind the selection
            DEER_CHECK_CUDA(cudaEventRecord(copy_ev, st), "record result event");
            DEER_CHECK_CUDA(cudaStreamWaitEvent(copy_st, copy_ev, 0), "wait result event");
        }
        DEER_CHECK_CUDA(cudaMemcpyAsync(y_host, y, N * n * sizeof(float), cudaMemcpyDeviceToHost, copy_st ? copy_st : st),
                        "copy result to host");
        return DEER_OK;
    };
    // bodies_done > 0: y holds the iterate after that many bodies of the one-launch form, which has given up
    hs.iters = bodies_done;
    if (bodies_done & 1)
        DEER_CHECK_CUDA(cudaMemcpyAsync(w.yalt, y, N * n * sizeof(float), cudaMemcpyDeviceToDevice, st), "copy iterate");
    const bool one_launch = bodies_done == 0 && body_takes(n, m, flags);
    HostSlot slot(one_launch);
    bool u_done = false;                       // w.u holds the projected inputs
    bool ended_there = false;                  // the one-launch form ran to the end
    if (one_launch) {
        if ((rc = eval_one_launch(p, x, y0, B, T, tol, max_iter, w, buf, flags, st, &hs, slot.p, u_done, y_host && !copy_early, polled, copy_out)) != DEER_OK) return rc;
        ended_there = hs.done == BODY_DONE;
        if (burn_in) *burn_in = ended_there ? hs.burn : -hs.burn;      // what its boundaries needed; negative: it gave up, what it would have needed
    }
    if (!one_launch || hs.done != BODY_DONE) {
    const int k0 = hs.iters;                   // bodies that the one-launch form has done
    if (k0 > 0) flags |= DEER_FLAG_WARM_START;
    hs.done = 0;
    const bool fused_proj = cell_projects(n, m) && ((((uintptr_t)y | (uintptr_t)y0) & 15) == 0);

    ScanArgs a{};
    a.J = w.J; a.b = w.rhs; a.y0 = y0; a.y = y;
    a.B = B; a.T = T; a.n = n; a.reverse = 0;
    a.L = w.scan.L; a.nch = w.scan.nch;
    a.carA = w.scan.carA; a.carB = w.scan.carB; a.starts = w.scan.starts;
    a.st = w.st;
    // With the single-pass scan the last CTA of every scan takes the loop decision and the scan
    // leaves its flag words cleared: a body is two launches (cell, scan).
    const bool single = scan_is_single_pass(a, w.scan, flags) && (((uintptr_t)w.yalt) & 15) == 0;
    // n = 16, 32: the cell writes coefficient rows and the scan generates J_t itself, unless the caller
    // asks for materialised Jacobians
    const bool gen_J = single && (n == 16 || n == 32 || (n == 64 && !(flags & DEER_FLAG_TCGEN05))) &&
                       !(flags & DEER_FLAG_MATERIALIZE) && ((((uintptr_t)y | (uintptr_t)y0 | (uintptr_t)p->W_h) & 15) == 0);
    // ... and the iteration runs in its Newton-update form: the scan solves for the update from a zero
    // entering update (its linear solve may then be approximate: single TF32 chain products)
    if (gen_J) { a.Wh = p->W_h; a.residual = 1; a.y0 = nullptr; }
    apply_test_flags(a, flags);
    {
        StatusBlock init;
        memset(&init, 0, sizeof(init));
        init.ctl_mode = single ? 1 : 0;
        init.max_iter = max_iter;
        init.tol = tol;
        init.trace = w.trace;
        init.iters = k0;
        // one launch: status block, zero initial guess, cleared words of the single-pass scan
        EvalBeginArgs e{};
        if (!(flags & DEER_FLAG_WARM_START)) { e.y = y; e.ny = N * n; }
        if (single) {
            const OnePassWs &op = w.scan.op;
            const size_t tiles = (size_t)B * op.nch;
            e.flags = op.flags; e.nflags = tiles;
            e.starts = op.starts; e.nstarts = tiles * (size_t)n;
            if (onepass_ll_aggs(n)) { e.agg_words = (unsigned long long *)op.aggs; e.nagg_words = tiles * (size_t)(n * n + n); }
        }
        const size_t words = e.ny / 4 + e.nflags + e.nstarts + e.nagg_words;
        unsigned blocks = (unsigned)((words + 1023) / 1024);
        const unsigned cap = 4u * (unsigned)num_sms();
        if (blocks > cap) blocks = cap;
        if (blocks < 1u) blocks = 1u;
        DEER_KERNEL("eval_begin_kernel", st, eval_begin_kernel<<<blocks, 256, 0, st>>>(w.st, init, e));
    }
    const bool cell_proj = gen_J && coef_cell_projects(n, m, x);     // (n = 32: the coefficient cell contracts x W_i^T itself)
    if (!fused_proj && !cell_proj && !u_done && (rc = run_proj(p, x, w.u, N, st)) != DEER_OK) return rc;

    // Newton loop (App. B.1): bodies are enqueued ahead of the convergence test -- the decision at
    // the end of each body is taken on the device, and the kernels of bodies past the end return
    // at once -- so the host only synchronises once per group of bodies.
    int enq = k0, group = 4;
    for (;;) {
        int todo = max_iter - enq;
        if (todo > group) todo = group;
        for (int j = 0; j < todo; ++j, ++enq) {
            float *cur = buf[enq & 1], *nxt = buf[(enq + 1) & 1];
            CellArgs c{p->W_h, p->b_h, (fused_proj || cell_proj) ? nullptr : w.u, x, p->W_i, p->b_i, m, cur, y0, w.J, w.rhs, B, T, n, w.st,
                       gen_J ? 1 : 0, gen_J ? 1 : 0};
            if ((rc = run_cell(c, st)) != DEER_OK) return rc;
            a.y = nxt; a.yold = cur;
            if (single) {
                if ((rc = scan_onepass(a, w.scan.op, false, flags, st)) != DEER_OK) return rc;
            } else {
                if ((rc = scan_generic(a, st)) != DEER_OK) return rc;
                DEER_KERNEL("newton_control_kernel", st, newton_control_kernel<<<1, 1, 0, st>>>(w.st, tol, max_iter, w.trace));
            }
        }
        if ((rc = copy_out(false)) != DEER_OK) return rc;
        DEER_CHECK_CUDA(cudaMemcpyAsync(&hs, w.st, 32, cudaMemcpyDeviceToHost, st), "read status");
        DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
        if (hs.flags & FLAG_TIMEOUT) return DEER_ERR_DEVICE_TIMEOUT;
        if (hs.done || enq >= max_iter) break;
        group = 2;
    }
    if ((rc = copy_out(true)) != DEER_OK) return rc;
    }
    const int k = hs.iters;
    float e;
    memcpy(&e, &hs.err_last_bits, sizeof(float));
    if ((err_b || err_argmax) && k > 0) {
        // the last two iterates are still in the two buffers (before the result copy below); a zero guess may not have been
        // written out
        if (k == 1 && !(flags & DEER_FLAG_WARM_START)) DEER_CHECK_CUDA(cudaMemsetAsync(buf[0], 0, N * n * sizeof(float), st), "zero guess");
        std::vector<unsigned long long> keys((size_t)B);
        DEER_KERNEL("err_diag_kernel", st, err_diag_kernel<<<(unsigned)B, 256, 0, st>>>(buf[k & 1], buf[(k + 1) & 1], (size_t)T * n, w.diag));
        DEER_CHECK_CUDA(cudaMemcpyAsync(keys.data(), w.diag, sizeof(unsigned long long) * (size_t)B, cudaMemcpyDeviceToHost, st), "read diagnostics");
        DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
        unsigned long long best = 0ull;
        int best_b = 0;
        for (int b = 0; b < B; ++b) {
            const unsigned bits = (unsigned)(keys[b] >> 32);
            if (err_b) memcpy(&err_b[b], &bits, sizeof(float));
            if ((keys[b] >> 32) > (best >> 32) || b == 0) { best = keys[b]; best_b = b; }
        }
        if (err_argmax)
            *err_argmax = (unsigned long long)best_b * (unsigned long long)T * (unsigned long long)n +
                          (unsigned long long)(0xffffffffu - (unsigned)(best & 0xffffffffull));
    }
    if ((k & 1) && !y_host)
        DEER_CHECK_CUDA(cudaMemcpyAsync(y, w.yalt, N * n * sizeof(float), cudaMemcpyDeviceToDevice, st), "copy result");
    const bool trace_here = ended_there && slot.p && k <= HOST_TRACE;
    if (err_trace && k > 0 && trace_here) memcpy(err_trace, slot.p->trace, sizeof(float) * (size_t)k);
    if (err_trace && k > 0 && !trace_here)
        DEER_CHECK_CUDA(cudaMemcpyAsync(err_trace, w.trace, sizeof(float) * (size_t)(k < ERR_TRACE_CAP ? k : ERR_TRACE_CAP),
                                        cudaMemcpyDeviceToHost, st), "read trace");
    if (((k & 1) && !y_host) || (y_host && !copy_early && !copy_st) || (err_trace && !trace_here)) DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
    if (iters) *iters = k;
    if (err) *err = e;
    return eval_status(e, tol);
}

// cell VJP, parameter-gradient slices and dx in one pass (n, m in {1,2,4,8}); P = slices written
template <int N, int M>
static int launch_vjp_small_nm(const VjpSmallArgs &v, int *P, cudaStream_t st)
{
    constexpr int EPB = 256 / N;
    constexpr size_t SM = sizeof(float) * 256 * (3 * (M + 1) + 3 * (N + 1) + 1);
    int rc = opt_in_smem((const void *)vjp_small_kernel<N, M>, SM);
    if (rc != DEER_OK) return rc;
    const size_t total = (size_t)v.B * v.T;
    size_t blocks = (total + EPB - 1) / EPB;
    if (blocks > (size_t)WGRAD_P) blocks = WGRAD_P;
    *P = (int)blocks;
    DEER_KERNEL("vjp_small_kernel", st, (vjp_small_kernel<N, M><<<(unsigned)blocks, 256, SM, st>>>(v)));
    return DEER_OK;
}

template <int N>
static int launch_vjp_small_n(const VjpSmallArgs &v, int m, int *P, cudaStream_t st)
{
    switch (m) {
    case 1: return launch_vjp_small_nm<N, 1>(v, P, st);
    case 2: return launch_vjp_small_nm<N, 2>(v, P, st);
    case 4: return launch_vjp_small_nm<N, 4>(v, P, st);
    case 8: return launch_vjp_small_nm<N, 8>(v, P, st);
    default: return DEER_ERR_UNSUPPORTED_N;
    }
}

static int launch_vjp_small(const VjpSmallArgs &v, int n, int m, int *P, cudaStream_t st)
{
    switch (n) {
    case 1: return launch_vjp_small_n<1>(v, m, P, st);
    case 2: return launch_vjp_small_n<2>(v, m, P, st);
    case 4: return launch_vjp_small_n<4>(v, m, P, st);
    case 8: return launch_vjp_small_n<8>(v, m, P, st);
    default: return DEER_ERR_UNSUPPORTED_N;
    }
}

// do the waits of the call's dense product k run out (test aid)?
static int expire_product(int flags, int k) { return (flags & DEER_FLAG_EXPIRE_PRODUCT_WAITS << k) != 0; }

// gy_seq (or nullptr): dL/dy is gy_seq [B,n] at every step, and gy a buffer for what has to read it position by position
static int gru_vjp_impl(const deer_gru_params *p, const float *x, const float *y0, const float *y,
                        const float *gy, int B, int T, const deer_gru_grads *g, float *dx,
                        float *dy0, void *ws, size_t ws_bytes, int flags, cudaStream_t st, int burn_hint = 0, const float *gy_seq = nullptr)
{
    const int n = p->n, m = p->m, n3 = 3 * n;
    VjpWs w = carve_vjp(ws, B, T, n, m);
    int rc = check_ws(ws, ws_bytes, w.bytes);
    if (rc != DEER_OK) return rc;
    const size_t N = (size_t)B * T;
    // small n and m: the cell projects x itself and one kernel does the cell VJP, the slices of the
    // parameter-gradient reduction and dx (no u, dG_i, dG_h arrays)
    const bool small = cell_projects(n, m) && !(flags & DEER_FLAG_GENERIC) && y0 != nullptr &&
                       ((((uintptr_t)y | (uintptr_t)y0) & 15) == 0);
    const bool have_u = !adjoint_supported(n, m, false);
    BodyPlan plan{};
    // n = 64: 128 chains per tcgen05 tile; else sixteen per warp
    BodyPlan tplan{};
    const bool exact_flags = (flags & (DEER_FLAG_GENERIC | DEER_FLAG_MATERIALIZE | DEER_FLAG_TCGEN05 | DEER_FLAG_EXPIRE_WAITS)) != 0;
    // (where the evaluation gave up, no try is made below what it would have needed)
    auto worth = [&](const BodyPlan &q) { return std::max(-burn_hint, ADJ_BURN) <= adjoint_burn_cap(n, m, (long long)B * T, q.L); };
    const bool tile = !exact_flags && (((uintptr_t)y | (uintptr_t)y0 | (uintptr_t)gy | (uintptr_t)x | (uintptr_t)p->W_h | (uintptr_t)p->W_i | (uintptr_t)dx) & 15) == 0 &&
                      adjoint_tile_plan(&tplan, B, T, n, m) && worth(tplan);
    const bool lanes = small && !exact_flags && (((uintptr_t)gy) & 3) == 0 && rows_adjoint_plan(&plan, B, T, n, m, WGRAD_P);     // all in one launch
    const bool adj = lanes || (!tile && !(flags & (DEER_FLAG_GENERIC | DEER_FLAG_MATERIALIZE | DEER_FLAG_TCGEN05 | DEER_FLAG_EXPIRE_WAITS)) &&
                     adjoint_plan(&plan, B, T, n, m, have_u, nullptr, 1) && worth(plan));
    if ((adj && !lanes && (size_t)plan.edges > w.start_groups) || ((adj || tile) && (size_t)(tile ? tplan : plan).edges > w.edges))
        return DEER_ERR_WORKSPACE;
    DEER_CHECK_CUDA(cudaMemsetAsync(w.st, 0, sizeof(StatusBlock) + (adj || tile ? (size_t)(tile ? tplan : plan).edges * sizeof(unsigned) : 0), st), "memset status");
    auto fill_gy = [&](const StatusBlock *done) -> int {
        DEER_KERNEL("broadcast_gy_kernel", st, broadcast_gy_kernel<<<dim3((unsigned)std::min((size_t)64, ((size_t)T * n + 1023) / 1024), B), 256, 0, st>>>(gy_seq, const_cast<float *>(gy), T, n, done));
        return DEER_OK;
    };
    if (gy_seq && !tile && (rc = fill_gy(nullptr)) != DEER_OK) return rc;
    // The contractions behind the adjoint in one pass, which takes packed rows: four stores of an adjoint step instead of six, a third
    // less to write (us per gradient, two arrays / packed: n = m = 32, 1.6e6 positions 1298 / 1262; n = 16, 960,000 614 / 590; n =
    // 20, 320,000 520 / 496; n = 48 718 / 730, whose adjoint spills: up to n = 32).  An adjoint that gives up leaves two arrays.
    GradTileArgs ga{};
    ga.dGi = w.dGi; ga.dGh = w.dGh;
    ga.x = x; ga.y = y; ga.y0 = y0; ga.W_i = p->W_i; ga.dx = dx;
    ga.slices = w.partial;
    ga.N = (int)N; ga.T = T; ga.n = n; ga.m = m;
    ga.expire = expire_product(flags, 0);
    ga.st = w.st;
    const bool one_pass = !(flags & DEER_FLAG_GENERIC) && N < 0x7fff0000u &&
                          grad_tile_suits(ga, (size_t)(w.partial2 - w.partial) + (size_t)WGRAD_P * n3 * (std::max(m, n) + 1));
    const bool packed = tile || (adj && !lanes && !small && one_pass && n <= 32);
    if (packed) ga.packed = w.st;
    const StatusBlock *unless = nullptr;       // set: the launches that take it do nothing where the adjoint launch has done the work
    if (adj || tile) {
        if (!tile && !lanes && have_u && (rc = run_proj(p, x, w.u, N, st)) != DEER_OK) return rc;
        AdjArgs a{};
        a.h0 = BodyHead{p->W_i, p->W_h, p->b_i, p->b_h, 1, 0, 0};
        a.x = x; a.u = !tile && !lanes && have_u ? w.u : nullptr; a.y0 = y0; a.y = y; a.gy = gy; a.gy_seq = tile ? gy_seq : nullptr;
        a.lam = small ? w.lam : nullptr; a.dGi = w.dGi; a.dGh = w.dGh; a.packed = packed ? 1 : 0;
        a.dy0 = dy0; a.dy0_by_head = 1;
        a.B = B; a.T = T; a.n = n; a.m = m; a.H = 1; a.L = tile ? tplan.L : plan.L;
        a.eta = ADJ_ETA;
        a.expire = (flags & DEER_FLAG_EXPIRE_BODY_WAITS) != 0;
        a.st = w.st; a.edge = w.edge; a.edge_flag = w.edge_flag; a.starts = tile ? w.J : w.starts;
        // (small cells: one try, the passes behind it are cheap)
        a.burn = !lanes && burn_hint > ADJ_BURN && burn_hint <= adjoint_burn_cap(n, m, (long long)B * T, a.L) ? burn_hint : ADJ_BURN;
        a.burn_cap = lanes ? 0 : adjoint_burn_cap(n, m, (long long)B * T, a.L);
        for (int k = 0; k < (lanes ? 1 : ADJ_TRIES); ++k) {
            if ((rc = tile ? launch_adjoint_tile(a, tplan, st) : lanes ? launch_rows_adjoint(a, plan, w.partial, w.partial2, dx, st) : launch_newton_adjoint(a, plan, st)) != DEER_OK) return rc;
        }
        unless = w.st;
        if (gy_seq && tile && (rc = fill_gy(unless)) != DEER_OK) return rc;
    }
    if (!small && !(adj && !lanes && have_u) && (rc = run_proj(p, x, w.u, N, st, unless)) != DEER_OK) return rc;
    ScanArgs a{};
    a.J = w.J; a.b = gy; a.y0 = nullptr; a.y = w.lam; a.yold = nullptr;
    a.B = B; a.T = T; a.n = n; a.reverse = 1;
    a.L = w.scan.L; a.nch = w.scan.nch;
    a.carA = w.scan.carA; a.carB = w.scan.carB; a.starts = w.scan.starts;
    a.st = w.st;
    // n = 16, 32: coefficient rows instead of Jacobians, J_{t+1}^T built in the reverse scan (as in the evaluation)
    const bool gen_J = (n == 16 || n == 32) && !(flags & DEER_FLAG_MATERIALIZE) && scan_is_single_pass(a, w.scan, flags) &&
                       ((((uintptr_t)y | (uintptr_t)y0 | (uintptr_t)p->W_h) & 15) == 0);
    if (gen_J) a.Wh = p->W_h;
    CellArgs c{p->W_h, p->b_h, small ? nullptr : w.u, x, p->W_i, p->b_i, m, y, y0, w.J, nullptr, B, T, n, unless,
               gen_J ? 1 : 0};
    if ((rc = run_cell(c, st)) != DEER_OK) return rc;
    if ((rc = run_scan(a, w.scan, flags, st, true, unless == nullptr)) != DEER_OK) return rc;

    if (small) {
        VjpSmallArgs v{p->W_h, p->b_h, p->W_i, p->b_i, x, y, y0, w.lam, dx, w.partial, w.partial2, B, T, lanes ? unless : nullptr};
        int P = 0;
        if ((rc = launch_vjp_small(v, n, m, &P, st)) != DEER_OK) return rc;
        const int oi = n3 * (m + 1), oh = n3 * (n + 1);
        DEER_KERNEL("wgrad_final_kernel", st, wgrad_final2_kernel<<<(oi + oh + 7) / 8, 256, 0, st>>>(w.partial, w.partial2, P, lanes ? unless : nullptr, plan.max_ctas, n3, m, n, g->dW_i, g->db_i, g->dW_h, g->db_h));
        if (dy0) {
            DEER_KERNEL("vjp_dy0_kernel", st, vjp_dy0_kernel<<<(B * n + 127) / 128, 128, 0, st>>>(w.J, w.lam, dy0, B, T, n, unless));
        }
        return DEER_OK;
    }
    {
        VjpArgs v{p->W_h, p->b_h, w.u, y, y0, w.lam, w.dGi, w.dGh, B, T, n, unless};
        const bool aligned = (((uintptr_t)y | (uintptr_t)y0) & 15) == 0;
        if (aligned && (n == 16 || n == 32 || n == 64)) {
            if ((rc = launch_vjp_cell_wide(v, st)) != DEER_OK) return rc;
        } else {
            size_t sm = sizeof(float) * (3 * n * (n + 1) + 3 * n);
            if ((rc = opt_in_smem((const void *)vjp_cell_kernel, sm)) != DEER_OK) return rc;
            int epb = 256 / n;
            unsigned blocks = (unsigned)((N + epb - 1) / epb);
            DEER_KERNEL("vjp_cell_kernel", st, vjp_cell_kernel<<<blocks, 256, sm, st>>>(v));
        }
    }
    const int P = (int)(N < (size_t)WGRAD_P ? N : (size_t)WGRAD_P);
    if (tile && !one_pass) return DEER_ERR_UNSUPPORTED_N;      // (never: packed rows are of n = 64, m <= 64, aligned)
    if (one_pass && (rc = launch_grad_tile(ga, g->dW_i, g->dW_h, g->db_i, g->db_h, st)) != DEER_OK) return rc;
    for (int side = 0; side < 2 && !one_pass; ++side) {
        WgradArgs wa{};
        wa.dG = side == 0 ? w.dGi : w.dGh;
        wa.V = side == 0 ? x : y;
        wa.y0 = y0;
        wa.shifted = side;
        wa.T = T; wa.n3 = n3; wa.K = side == 0 ? m : n;
        wa.N = N; wa.slice = (N + P - 1) / P;
        wa.partial = w.partial;
        int outs = n3 * (wa.K + 1);
        if (n3 <= 32 && wa.K <= 8) {
            DEER_KERNEL("wgrad_small_kernel", st, wgrad_small_kernel<<<P, 256, 0, st>>>(wa));
        } else if (n3 <= 192) {
            const bool aligned16 = ((((uintptr_t)wa.dG | (uintptr_t)wa.V | (uintptr_t)wa.y0) & 15) == 0) && n3 % 4 == 0 && wa.K % 4 == 0;
            if (aligned16) {
                const size_t sm = wgrad_staged_smem(n3);
                if ((rc = opt_in_smem((const void *)wgrad_mma_staged_kernel, sm)) != DEER_OK) return rc;
                DEER_KERNEL("wgrad_mma_kernel", st, wgrad_mma_staged_kernel<<<dim3(P, (wa.K + 63) / 64), 32 * ((n3 + 15) / 16), sm, st>>>(wa));
            } else {
                DEER_KERNEL("wgrad_mma_kernel", st, wgrad_mma_kernel<<<dim3(P, (wa.K + 63) / 64), 32 * ((n3 + 15) / 16), 0, st>>>(wa));
            }
        } else {
            int tile = 32;
            while (tile > 1 && sizeof(float) * tile * (size_t)(n3 + wa.K + 1) > 160 * 1024) tile >>= 1;
            wa.tile = tile;
            size_t sm = sizeof(float) * tile * (size_t)(n3 + wa.K + 1);
            if ((rc = opt_in_smem((const void *)wgrad_partial_kernel, sm)) != DEER_OK) return rc;
            dim3 grid(P, (outs + 255) / 256);
            DEER_KERNEL("wgrad_partial_kernel", st, wgrad_partial_kernel<<<grid, 256, sm, st>>>(wa));
        }
        DEER_KERNEL("wgrad_final_kernel", st, wgrad_final_kernel<<<(outs + 7) / 8, 256, 0, st>>>(w.partial, P, n3, wa.K,
                                                                side == 0 ? g->dW_i : g->dW_h,
                                                                side == 0 ? g->db_i : g->db_h));
    }
    if (dx && !one_pass) {
        if (m >= 32 && m <= 256) {
            if ((rc = run_affine(w.dGi, p->W_i, nullptr, dx, N, n3, m, 1, st)) != DEER_OK) return rc;
        } else {
            size_t total = N * (size_t)m;
            DEER_KERNEL("vjp_dx_kernel", st, vjp_dx_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(w.dGi, p->W_i, dx, N, m, n3));
        }
    }
    if (dy0) {
        if (gen_J) {
            DEER_KERNEL("vjp_dy0_coef_kernel", st, vjp_dy0_coef_kernel<<<(B * n + 127) / 128, 128, 0, st>>>(w.J, p->W_h, w.lam, dy0, B, T, n, unless));
        } else {
            DEER_KERNEL("vjp_dy0_kernel", st, vjp_dy0_kernel<<<(B * n + 127) / 128, 128, 0, st>>>(w.J, w.lam, dy0, B, T, n, unless));
        }
    }
    return DEER_OK;
}

// ---------------------------------------------------------------- built-in scratch (no-alloc entry point)
// In host code `g_noalloc_scratch` is only a handle for the runtime, not a device address: the
// address a kernel can use comes from cudaGetSymbolAddress, looked up once per device.
static __device__ __align__(256) unsigned char g_noalloc_scratch[DEER_NOALLOC_SCRATCH_BYTES];

static std::mutex g_noalloc_mu;
static void *g_noalloc_ptr[64] = {nullptr};

static int noalloc_scratch_for_current_device(void **out)
{
    int dev = -1;
    DEER_CHECK_CUDA(cudaGetDevice(&dev), "cudaGetDevice");
    if (dev < 0 || dev >= 64) { snprintf(t_err, sizeof(t_err), "device index %d out of range", dev); return DEER_ERR_CUDA; }
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        DEER_CHECK_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch), "cudaGetSymbolAddress(scratch)");
        if (!p || ((uintptr_t)p & 255) != 0) { snprintf(t_err, sizeof(t_err), "built-in scratch misaligned"); return DEER_ERR_CUDA; }
        g_noalloc_ptr[dev] = p;
    }
    *out = g_noalloc_ptr[dev];
    return DEER_OK;
}

}  // namespace deer

using namespace deer;

// ---------------------------------------------------------------- exported C ABI
extern "C" {

size_t deer_workspace_bytes(int op, int B, int T, int n, int m, int flags)
{
    (void)flags;
    if (op == DEER_OP_SCAN || op == DEER_OP_ODE) m = 1;
    if (!valid_sizes(B, T, n, m) || !supported(n, m)) return 0;
    switch (op) {
    case DEER_OP_EVAL: return carve_eval(nullptr, B, T, n, m).bytes;
    case DEER_OP_SCAN: return carve_scan_only(nullptr, B, T, n).bytes;
    case DEER_OP_VJP: return carve_vjp(nullptr, B, T, n, m).bytes;
    case DEER_OP_CLASSIFIER: return carve_cls(nullptr, B, T, n, m, 64).bytes;
    case DEER_OP_ODE: return n <= ODE_MAX_N ? carve_ode(nullptr, B, T, n).bytes : 0;
    case DEER_OP_LSTM: return supported(2 * n, m) ? carve_lstm(nullptr, B, T, n).bytes : 0;
    default: return 0;
    }
}

int deer_linrec_scan(const float *J, const float *b, const float *y0, int B, int T, int n,
                     int reverse, float *y, void *ws, size_t ws_bytes, int flags, void *stream)
{
    if (!J || !b || !y || B <= 0 || T <= 0 || n <= 0) return DEER_ERR_INVALID_ARG;
    if (!supported(n, 1)) return DEER_ERR_UNSUPPORTED_N;
    if (!valid_sizes(B, T, n, 1)) return DEER_ERR_INVALID_ARG;
    return linrec_scan_impl(J, b, y0, B, T, n, reverse, y, ws, ws_bytes, flags, (cudaStream_t)stream);
}

int deer_gru_eval(const deer_gru_params *p, const float *x, const float *y0, int B, int T, float tol,
                  int max_iter, float *y, int *iters, float *err, float *err_trace, void *ws,
                  size_t ws_bytes, int flags, void *stream)
{
    if (!p || !x || !y0 || !y || !p->W_i || !p->W_h || !p->b_i || !p->b_h) return DEER_ERR_INVALID_ARG;
    if (B <= 0 || T <= 0 || p->n <= 0 || p->m <= 0 || max_iter < 1 || tol != tol) return DEER_ERR_INVALID_ARG;
    if (!supported(p->n, p->m)) return DEER_ERR_UNSUPPORTED_N;
    if (!valid_sizes(B, T, p->n, p->m)) return DEER_ERR_INVALID_ARG;
    return gru_eval_impl(p, x, y0, B, T, tol, max_iter, y, iters, err, err_trace, ws, ws_bytes, flags,
                         (cudaStream_t)stream);
}

int deer_gru_eval_diag(const deer_gru_params *p, const float *x, const float *y0, int B, int T, float tol,
                       int max_iter, float *y, int *iters, float *err, float *err_trace, float *err_b,
                       unsigned long long *err_argmax, void *ws, size_t ws_bytes, int flags, void *stream)
{
    if (!p || !x || !y0 || !y || !p->W_i || !p->W_h || !p->b_i || !p->b_h) return DEER_ERR_INVALID_ARG;
    if (B <= 0 || T <= 0 || p->n <= 0 || p->m <= 0 || max_iter < 1 || tol != tol) return DEER_ERR_INVALID_ARG;
    if (!supported(p->n, p->m)) return DEER_ERR_UNSUPPORTED_N;
    if (!valid_sizes(B, T, p->n, p->m)) return DEER_ERR_INVALID_ARG;
    if ((unsigned long long)T * (unsigned long long)p->n > 0xffffffffull) return DEER_ERR_INVALID_ARG;
    return gru_eval_impl(p, x, y0, B, T, tol, max_iter, y, iters, err, err_trace, ws, ws_bytes, flags,
                         (cudaStream_t)stream, nullptr, err_b, err_argmax);
}

// Copy streams and events of the pipelined host call, one set per device, made on first use.
struct HostPipe {
    cudaStream_t h2d = nullptr, d2h = nullptr;
    cudaEvent_t ev_in = nullptr, ev_sel = nullptr, ev_out = nullptr, ev_chunk[DEER_HOST_MAX_CHUNKS] = {};
    bool ready = false;
    std::mutex mu;
};
static HostPipe g_host_pipe[MAX_DEVICES];

static int host_pipe_for_current_device(HostPipe **out)
{
    int dev = 0;
    DEER_CHECK_CUDA(cudaGetDevice(&dev), "cudaGetDevice");
    if (dev < 0 || dev >= MAX_DEVICES) return DEER_ERR_INVALID_ARG;
    HostPipe &hp = g_host_pipe[dev];
    if (!hp.ready) {
        DEER_CHECK_CUDA(cudaStreamCreateWithFlags(&hp.h2d, cudaStreamNonBlocking), "create copy stream");
        DEER_CHECK_CUDA(cudaStreamCreateWithFlags(&hp.d2h, cudaStreamNonBlocking), "create copy stream");
        DEER_CHECK_CUDA(cudaEventCreateWithFlags(&hp.ev_in, cudaEventDisableTiming), "create event");
        DEER_CHECK_CUDA(cudaEventCreateWithFlags(&hp.ev_sel, cudaEventDisableTiming), "create event");
        DEER_CHECK_CUDA(cudaEventCreateWithFlags(&hp.ev_out, cudaEventDisableTiming), "create event");
        for (int c = 0; c < DEER_HOST_MAX_CHUNKS; ++c)
            DEER_CHECK_CUDA(cudaEventCreateWithFlags(&hp.ev_chunk[c], cudaEventDisableTiming), "create event");
        hp.ready = true;
    }
    *out = &hp;
    return DEER_OK;
}

int deer_gru_eval_host_chunks(int B, int T, int *first)
{
    if (B <= 0 || T <= 0) return 0;
    // chunks of about 2^19 positions: long enough to fill the GPU, short enough that the first copy in and the last
    // copy out (the two that nothing hides) are a small part of the call (config 3: three chunks measured best of 1 ... 8)
    const long long N = (long long)B * T;
    long long nc = (N + 262144) / 524288;
    if (nc > DEER_HOST_MAX_CHUNKS) nc = DEER_HOST_MAX_CHUNKS;
    if (nc > B) nc = B;
    if (nc < 1) nc = 1;
    if (first) {
        first[0] = 0;
        for (int k = 1; k < (int)nc; ++k) {
            // equal chunks for two; from three on the first and the last weigh half: their copies are the exposed ones
            // (config 3: 4, 8, 4 sequences measured 9.1 ms per call against 9.65 for 6, 6, 4)
            long long b = nc < 3 ? ((long long)B * k + nc - 1) / nc
                                 : ((long long)B * (2 * k - 1) + (nc - 1)) / (2 * (nc - 1));
            const long long lo = first[k - 1] + 1, hi = B - (nc - k);
            first[k] = (int)(b < lo ? lo : b > hi ? hi : b);
        }
        first[nc] = B;
    }
    return (int)nc;
}

int deer_gru_eval_host_chunk(int B, int T)
{
    int first[DEER_HOST_MAX_CHUNKS + 1];
    const int nc = deer_gru_eval_host_chunks(B, T, first);
    int big = 0;
    for (int c = 0; c < nc; ++c) big = std::max(big, first[c + 1] - first[c]);
    return big;
}

int deer_gru_eval_host(const deer_gru_params *p, const float *x_host, const float *y0, int B, int T, float tol,
                       int max_iter, float *y_host, int *iters, float *err, float *x_dev, float *y_dev,
                       void *ws, size_t ws_bytes, int flags, void *stream)
{
    if (!p || !x_host || !y0 || !y_host || !x_dev || !y_dev || !p->W_i || !p->W_h || !p->b_i || !p->b_h)
        return DEER_ERR_INVALID_ARG;
    if (B <= 0 || T <= 0 || p->n <= 0 || p->m <= 0 || max_iter < 1 || tol != tol) return DEER_ERR_INVALID_ARG;
    if (!supported(p->n, p->m)) return DEER_ERR_UNSUPPORTED_N;
    if (!valid_sizes(B, T, p->n, p->m)) return DEER_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    int bnd[DEER_HOST_MAX_CHUNKS + 1];
    const int nc = deer_gru_eval_host_chunks(B, T, bnd);
    if (nc <= 1) {
        DEER_CHECK_CUDA(cudaMemcpyAsync(x_dev, x_host, sizeof(float) * (size_t)B * T * p->m, cudaMemcpyHostToDevice, st),
                        "copy x to the device");
        return gru_eval_impl(p, x_dev, y0, B, T, tol, max_iter, y_dev, iters, err, nullptr, ws, ws_bytes, flags, st, y_host);
    }
    // Sequences are independent (the batch is a map over sequences), so the batch is evaluated in chunks of sequences,
    // each with its own Newton loop: chunk c + 1 arrives and chunk c - 1 leaves while chunk c is evaluated.
    {
        EvalWs wfull = carve_eval(ws, B, T, p->n, p->m);       // (the caller sized ws for the whole batch: checked as documented)
        int rc = check_ws(ws, ws_bytes, wfull.bytes);
        if (rc != DEER_OK) return rc;
    }
    HostPipe *hp = nullptr;
    int rc = host_pipe_for_current_device(&hp);
    if (rc != DEER_OK) return rc;
    std::lock_guard<std::mutex> lk(hp->mu);
    const size_t xs = (size_t)T * p->m, ys = (size_t)T * p->n;
    DEER_CHECK_CUDA(cudaEventRecord(hp->ev_in, st), "record entry event");
    DEER_CHECK_CUDA(cudaStreamWaitEvent(hp->h2d, hp->ev_in, 0), "wait entry event");
    DEER_CHECK_CUDA(cudaStreamWaitEvent(hp->d2h, hp->ev_in, 0), "wait entry event");
    for (int c = 0; c < nc; ++c) {
        const int b0 = bnd[c], bn = bnd[c + 1] - b0;
        DEER_CHECK_CUDA(cudaMemcpyAsync(x_dev + b0 * xs, x_host + b0 * xs, sizeof(float) * bn * xs, cudaMemcpyHostToDevice, hp->h2d),
                        "copy x to the device");
        DEER_CHECK_CUDA(cudaEventRecord(hp->ev_chunk[c], hp->h2d), "record chunk event");
    }
    int status = DEER_OK, k_max = 0;
    float e_max = 0.0f;
    for (int c = 0; c < nc; ++c) {
        const int b0 = bnd[c], bn = bnd[c + 1] - b0;
        DEER_CHECK_CUDA(cudaStreamWaitEvent(st, hp->ev_chunk[c], 0), "wait chunk event");
        int k = 0;
        float e = 0.0f;
        rc = gru_eval_impl(p, x_dev + b0 * xs, y0 + (size_t)b0 * p->n, bn, T, tol, max_iter, y_dev + b0 * ys, &k, &e, nullptr,
                           ws, ws_bytes, flags, st, y_host + b0 * ys, nullptr, nullptr, hp->d2h, hp->ev_sel);
        if (rc < 0) { cudaStreamSynchronize(hp->h2d); cudaStreamSynchronize(hp->d2h); return rc; }
        if (k > k_max) k_max = k;
        if (!(e <= e_max)) e_max = e;                              // (keeps a NaN)
        if (rc == DEER_NONFINITE || (rc == DEER_NOT_CONVERGED && status == DEER_OK)) status = rc;
    }
    DEER_CHECK_CUDA(cudaEventRecord(hp->ev_out, hp->d2h), "record exit event");
    DEER_CHECK_CUDA(cudaStreamWaitEvent(st, hp->ev_out, 0), "wait exit event");
    DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
    if (iters) *iters = k_max;
    if (err) *err = e_max;
    return status;
}

int deer_gru_vjp(const deer_gru_params *p, const float *x, const float *y0, const float *y,
                 const float *gy, int B, int T, const deer_gru_grads *g, float *dx, float *dy0,
                 void *ws, size_t ws_bytes, int flags, void *stream)
{
    if (!p || !x || !y0 || !y || !gy || !g || !p->W_i || !p->W_h || !p->b_i || !p->b_h)
        return DEER_ERR_INVALID_ARG;
    if (!g->dW_i || !g->dW_h || !g->db_i || !g->db_h) return DEER_ERR_INVALID_ARG;
    if (B <= 0 || T <= 0 || p->n <= 0 || p->m <= 0) return DEER_ERR_INVALID_ARG;
    if (!supported(p->n, p->m)) return DEER_ERR_UNSUPPORTED_N;
    if (!valid_sizes(B, T, p->n, p->m)) return DEER_ERR_INVALID_ARG;
    return gru_vjp_impl(p, x, y0, y, gy, B, T, g, dx, dy0, ws, ws_bytes, flags, (cudaStream_t)stream);
}

// The burn-in that a gradient's boundaries need, from the one that the bodies of the same trajectory would have needed for eta
// (0: they do not tell; negative: the evaluation gave up): it goes with the logarithm of the accuracy asked for.  (Needed / told
// so, without the tenth and the two, of twelve first layers of 64: 47 / 42, 45 / 45, 39 / 40, 43 / 48, 55 / 52, 46 / 51, 46 / 43,
// 48 / 53, 40 / 41, 39 / 38, 42 / 43; a try that is too short costs all of its 75 steps.)
static int adjoint_burn_hint(int burn, int n, float tol)
{
    if (burn <= 0 && -burn <= body_first_burn(n, tol)) return 0;
    const float to = logf(0.5f * ADJ_ETA) / logf(0.5f * body_eta(n, tol));
    return (int)fmaxf(-1e6f, fminf(1e6f, burn > 0 ? 1.1f * to * (float)burn + 2.0f : to * (float)burn));
}

int deer_gru_classifier_step(const deer_gru_params *l1, const deer_gru_params *l2, const float *W_o,
                             const float *b_o, int ncls, const float *x, const int *labels, int B,
                             int T, float tol, int max_iter, float *loss, int *iters,
                             const deer_gru_grads *g1, const deer_gru_grads *g2, float *dW_o,
                             float *db_o, void *ws, size_t ws_bytes, int flags, void *stream)
{
    if (!l1 || !l2 || !W_o || !b_o || !x || !labels || !loss || !g1 || !g2 || !dW_o || !db_o)
        return DEER_ERR_INVALID_ARG;
    if (B <= 0 || T <= 0 || ncls < 1 || ncls > 64 || max_iter < 1 || tol != tol) return DEER_ERR_INVALID_ARG;
    if (l1->n != l2->n || l2->m != l1->n) return DEER_ERR_INVALID_ARG;
    if (!supported(l1->n, l1->m) || !supported(l2->n, l2->m)) return DEER_ERR_UNSUPPORTED_N;
    if (B * ncls > 4096 || B * l1->n > 65536) return DEER_ERR_INVALID_ARG;
    const int n = l1->n, m = l1->m;
    cudaStream_t st = (cudaStream_t)stream;
    ClsWs w = carve_cls(ws, B, T, n, m, 64);
    int rc = check_ws(ws, ws_bytes, w.bytes);
    if (rc != DEER_OK) return rc;
    for (const deer_gru_params *l : {l1, l2})
        if (!l->W_i || !l->W_h || !l->b_i || !l->b_h || l->m <= 0 || !valid_sizes(B, T, l->n, l->m)) return DEER_ERR_INVALID_ARG;
    for (const deer_gru_grads *g : {g1, g2})
        if (!g->dW_i || !g->dW_h || !g->db_i || !g->db_h) return DEER_ERR_INVALID_ARG;
    // zero initial states live at the head of gyB until the backward pass needs it
    float *zero0 = w.gyB;
    DEER_CHECK_CUDA(cudaMemsetAsync(zero0, 0, (size_t)B * n * sizeof(float), st), "memset y0");
    int it[2] = {0, 0};
    int burn1 = 0, burn2 = 0;
    int s1 = gru_eval_impl(l1, x, zero0, B, T, tol, max_iter, w.y1, &it[0], nullptr, nullptr, w.inner,
                           w.inner_bytes, flags, st, nullptr, nullptr, nullptr, nullptr, nullptr, 0, &burn1);
    if (s1 < 0) return s1;
    int s2 = gru_eval_impl(l2, w.y1, zero0, B, T, tol, max_iter, w.y2, &it[1], nullptr, nullptr,
                           w.inner, w.inner_bytes, flags, st, nullptr, nullptr, nullptr, nullptr, nullptr, 0, &burn2);
    if (s2 < 0) return s2;
    if (iters) { iters[0] = it[0]; iters[1] = it[1]; }
    int seg_len = (T + POOL_SEGS - 1) / POOL_SEGS;
    DEER_KERNEL("pool_partial_kernel", st, pool_partial_kernel<<<dim3(POOL_SEGS, B), n, 0, st>>>(w.y2, T, n, seg_len, w.pool_partial));
    DEER_KERNEL("head_kernel", st, head_kernel<<<1, HEAD_THREADS, 0, st>>>(w.pool_partial, POOL_SEGS, B, T, n, ncls, W_o, b_o, labels,
                                   w.pooled, w.dlog, w.gpool, dW_o, db_o, w.loss));
    // zero states again (gyB is about to be overwritten by dx of layer 2): use pooled' neighbour
    float *zero1 = w.pool_partial;   // >= B*n floats, no longer needed
    DEER_CHECK_CUDA(cudaMemsetAsync(zero1, 0, (size_t)B * n * sizeof(float), st), "memset y0");
    // the backward passes are asynchronous and share one status block: the flags word of each is
    // saved beside the loss before the next call clears it, and both are read after the final sync
    const unsigned *vflags = &reinterpret_cast<const StatusBlock *>(w.inner)->flags;
    rc = gru_vjp_impl(l2, w.y1, zero1, w.y2, w.gyA, B, T, g2, w.gyB, nullptr, w.inner, w.inner_bytes,
                      flags, st, adjoint_burn_hint(burn2, n, tol), w.gpool);
    if (rc != DEER_OK) return rc;
    DEER_CHECK_CUDA(cudaMemcpyAsync(w.loss + 1, vflags, sizeof(unsigned), cudaMemcpyDeviceToDevice, st), "save status");
    rc = gru_vjp_impl(l1, x, zero1, w.y1, w.gyB, B, T, g1, nullptr, nullptr, w.inner, w.inner_bytes,
                      flags, st, adjoint_burn_hint(burn1, n, tol));
    if (rc != DEER_OK) return rc;
    DEER_CHECK_CUDA(cudaMemcpyAsync(w.loss + 2, vflags, sizeof(unsigned), cudaMemcpyDeviceToDevice, st), "save status");
    float tail[3];
    DEER_CHECK_CUDA(cudaMemcpyAsync(tail, w.loss, sizeof(tail), cudaMemcpyDeviceToHost, st), "read loss");
    DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
    unsigned f1, f2;
    memcpy(&f1, &tail[1], sizeof(unsigned)); memcpy(&f2, &tail[2], sizeof(unsigned));
    if ((f1 | f2) & FLAG_TIMEOUT) return DEER_ERR_DEVICE_TIMEOUT;
    *loss = tail[0];
    return s1 > s2 ? s1 : s2;
}

int deer_gru_jvp(const deer_gru_params *p, const deer_gru_params *dp, const float *x, const float *dx, const float *y0,
                 const float *dy0, const float *y, int B, int T, float *dy, void *ws, size_t ws_bytes, int flags,
                 void *stream)
{
    if (!p || !x || !y0 || !y || !dy || !p->W_i || !p->W_h || !p->b_i || !p->b_h) return DEER_ERR_INVALID_ARG;
    if (B <= 0 || T <= 0 || p->n <= 0 || p->m <= 0) return DEER_ERR_INVALID_ARG;
    if (dp && (dp->n != p->n || dp->m != p->m)) return DEER_ERR_INVALID_ARG;
    if (!supported(p->n, p->m)) return DEER_ERR_UNSUPPORTED_N;
    if (!valid_sizes(B, T, p->n, p->m)) return DEER_ERR_INVALID_ARG;
    const int n = p->n, m = p->m, n3 = 3 * n;
    cudaStream_t st = (cudaStream_t)stream;
    // the gradient's workspace layout holds what is needed: u, J, and three [B,T,3n] / [B,T,n] arrays
    VjpWs w = carve_vjp(ws, B, T, n, m);
    int rc = check_ws(ws, ws_bytes, w.bytes);
    if (rc != DEER_OK) return rc;
    const size_t N = (size_t)B * T;
    DEER_CHECK_CUDA(cudaMemsetAsync(w.st, 0, sizeof(StatusBlock), st), "memset status");
    if ((rc = run_proj(p, x, w.u, N, st)) != DEER_OK) return rc;
    // du1 = x dW_i^T + db_i ;  du2 = dx W_i^T
    float *du1 = nullptr, *du2 = nullptr;
    const bool have_di = dp && (dp->W_i || dp->b_i);
    if (have_di) {
        if (!dp->W_i || !dp->b_i) return DEER_ERR_INVALID_ARG;       // the input-side pair comes together
        deer_gru_params q = *p;
        q.W_i = dp->W_i; q.b_i = dp->b_i;
        du1 = w.dGi;
        if ((rc = run_proj(&q, x, du1, N, st)) != DEER_OK) return rc;
    }
    if (dx) {
        du2 = w.dGh;
        if ((rc = run_affine(dx, p->W_i, nullptr, du2, N, m, n3, 0, st)) != DEER_OK) return rc;
    }
    if (dp && ((dp->W_h == nullptr) != (dp->b_h == nullptr))) return DEER_ERR_INVALID_ARG;
    {
        JvpArgs j{p->W_h, p->b_h, dp ? dp->W_h : nullptr, dp ? dp->b_h : nullptr, w.u, du1, du2, y, y0, w.lam, B, T, n};
        const size_t sm = sizeof(float) * (6 * (size_t)n * (n + 1) + 6 * n);
        if ((rc = opt_in_smem((const void *)jvp_cell_kernel, sm)) != DEER_OK) return rc;
        const int epb = 256 / n;
        size_t blocks = (N + epb - 1) / epb;
        const size_t cap = (size_t)num_sms() * 8;
        if (blocks > cap) blocks = cap;
        DEER_KERNEL("jvp_cell_kernel", st, jvp_cell_kernel<<<(unsigned)blocks, 256, sm, st>>>(j));
    }
    // the Jacobians at the trajectory (exact: a one-shot solve), then dy = L_G^{-1}[df] from dy0 (Sec. 3.1.1)
    ScanArgs a{};
    a.J = w.J; a.b = w.lam; a.y0 = dy0; a.y = dy; a.yold = nullptr;
    a.B = B; a.T = T; a.n = n; a.reverse = 0;
    a.L = w.scan.L; a.nch = w.scan.nch;
    a.carA = w.scan.carA; a.carB = w.scan.carB; a.starts = w.scan.starts;
    a.st = w.st;
    CellArgs c{p->W_h, p->b_h, w.u, x, p->W_i, p->b_i, m, y, y0, w.J, nullptr, B, T, n, nullptr, 0, 0};
    if ((rc = run_cell(c, st)) != DEER_OK) return rc;
    return run_scan(a, w.scan, flags, st, true, true);
}

int deer_lstm_eval(const deer_lstm_params *p, const float *x, const float *s0, int B, int T, float tol, int max_iter,
                   float *s_out, int *iters, float *err, void *ws, size_t ws_bytes, int flags, void *stream)
{
    if (!p || !x || !s0 || !s_out || !p->W_i || !p->W_h || !p->b) return DEER_ERR_INVALID_ARG;
    if (B <= 0 || T <= 0 || p->k <= 0 || p->m <= 0 || max_iter < 1 || tol != tol) return DEER_ERR_INVALID_ARG;
    if (!supported(2 * p->k, p->m)) return DEER_ERR_UNSUPPORTED_N;
    if (!valid_sizes(B, T, 2 * p->k, p->m)) return DEER_ERR_INVALID_ARG;
    const int k = p->k, m = p->m, n = 2 * k;
    cudaStream_t st = (cudaStream_t)stream;
    LstmWs w = carve_lstm(ws, B, T, k);
    int rc = check_ws(ws, ws_bytes, w.bytes);
    if (rc != DEER_OK) return rc;
    const size_t N = (size_t)B * T;

    ScanArgs a{};
    a.J = w.J; a.b = w.rhs; a.y0 = s0; a.y = s_out;
    a.B = B; a.T = T; a.n = n; a.reverse = 0;
    a.L = w.scan.L; a.nch = w.scan.nch;
    a.carA = w.scan.carA; a.carB = w.scan.carB; a.starts = w.scan.starts;
    a.st = w.st;
    apply_test_flags(a, flags);
    const bool single = scan_is_single_pass(a, w.scan, flags) && (((uintptr_t)w.yalt) & 15) == 0;
    {
        StatusBlock init;
        memset(&init, 0, sizeof(init));
        init.ctl_mode = single ? 1 : 0;
        init.max_iter = max_iter;
        init.tol = tol;
        init.trace = w.trace;
        EvalBeginArgs e{};
        if (!(flags & DEER_FLAG_WARM_START)) { e.y = s_out; e.ny = N * n; }
        if (single) {
            const OnePassWs &op = w.scan.op;
            const size_t tiles = (size_t)B * op.nch;
            e.flags = op.flags; e.nflags = tiles;
            e.starts = op.starts; e.nstarts = tiles * (size_t)n;
            if (onepass_ll_aggs(n)) { e.agg_words = (unsigned long long *)op.aggs; e.nagg_words = tiles * (size_t)(n * n + n); }
        }
        const size_t words = e.ny / 4 + e.nflags + e.nstarts + e.nagg_words;
        unsigned blocks = (unsigned)((words + 1023) / 1024);
        const unsigned cap = 4u * (unsigned)num_sms();
        if (blocks > cap) blocks = cap;
        if (blocks < 1u) blocks = 1u;
        DEER_KERNEL("eval_begin_kernel", st, eval_begin_kernel<<<blocks, 256, 0, st>>>(w.st, init, e));
    }
    // u = x W_i^T + b  (4k outputs per position; iteration-invariant)
    if (sizeof(float) * ((size_t)m * 4 * k + (size_t)PROJ_PP * (m + 1)) <= 200 * 1024 && 4 * k <= 256) {
        if ((rc = run_affine(x, p->W_i, p->b, w.u, N, m, 4 * k, 0, st)) != DEER_OK) return rc;
    } else {
        const size_t total = N * (size_t)(4 * k);
        DEER_KERNEL("proj_kernel", st, proj_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(x, p->W_i, p->b, w.u, N, m, 4 * k, nullptr));
    }
    const size_t sm = sizeof(float) * 4 * (size_t)k * (k + 1);
    if ((rc = opt_in_smem((const void *)lstm_cell_kernel, sm)) != DEER_OK) return rc;
    const int threads = 256 / k * k;
    size_t cblocks = (N + (size_t)(256 / k) - 1) / (size_t)(256 / k);
    if (cblocks > (size_t)num_sms() * 16) cblocks = (size_t)num_sms() * 16;

    float *buf[2] = {s_out, w.yalt};
    int enq = 0, group = 4;
    StatusBlock hs;
    for (;;) {
        int todo = max_iter - enq;
        if (todo > group) todo = group;
        for (int j = 0; j < todo; ++j, ++enq) {
            float *cur = buf[enq & 1], *nxt = buf[(enq + 1) & 1];
            LstmCellArgs c{p->W_h, w.u, cur, s0, w.J, w.rhs, B, T, k, w.st};
            DEER_KERNEL("lstm_cell_kernel", st, lstm_cell_kernel<<<(unsigned)cblocks, threads, sm, st>>>(c));
            a.y = nxt; a.yold = cur;
            if (single) {
                if ((rc = scan_onepass(a, w.scan.op, false, flags, st)) != DEER_OK) return rc;
            } else {
                if ((rc = scan_generic(a, st)) != DEER_OK) return rc;
                DEER_KERNEL("newton_control_kernel", st, newton_control_kernel<<<1, 1, 0, st>>>(w.st, tol, max_iter, w.trace));
            }
        }
        DEER_CHECK_CUDA(cudaMemcpyAsync(&hs, w.st, 32, cudaMemcpyDeviceToHost, st), "read status");
        DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
        if (hs.flags & FLAG_TIMEOUT) return DEER_ERR_DEVICE_TIMEOUT;
        if (hs.done || enq >= max_iter) break;
        group = 2;
    }
    const int kk = hs.iters;
    float e;
    memcpy(&e, &hs.err_last_bits, sizeof(float));
    if (kk & 1)
        DEER_CHECK_CUDA(cudaMemcpyAsync(s_out, w.yalt, N * n * sizeof(float), cudaMemcpyDeviceToDevice, st), "copy result");
    DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
    int status = DEER_OK;
    if (!isfinite(e)) status = DEER_NONFINITE;
    else if (e > tol && !(tol < 0.0f)) status = DEER_NOT_CONVERGED;
    if (iters) *iters = kk;
    if (err) *err = e;
    return status;
}

int deer_ode_linear_solve(const float *G, const float *z, const float *t, const float *y0, int B, int T, int n, float *y,
                          void *ws, size_t ws_bytes, int flags, void *stream)
{
    if (!G || !z || !t || !y0 || !y || B <= 0 || T <= 0 || n <= 0) return DEER_ERR_INVALID_ARG;
    if (n > ODE_MAX_N) return DEER_ERR_UNSUPPORTED_N;
    if (!valid_sizes(B, T, n, 1)) return DEER_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    OdeWs w = carve_ode(ws, B, T, n);
    int rc = check_ws(ws, ws_bytes, w.bytes);
    if (rc != DEER_OK) return rc;
    DEER_CHECK_CUDA(cudaMemsetAsync(w.st, 0, sizeof(StatusBlock), st), "memset status");
    {
        const size_t sm = sizeof(float) * 3 * (size_t)(n + 1) * (n + 1) * ODE_THREADS;
        if ((rc = opt_in_smem((const void *)ode_discretise_kernel, sm)) != DEER_OK) return rc;
        size_t blocks = ((size_t)B * T + ODE_THREADS - 1) / ODE_THREADS;
        const size_t cap = (size_t)num_sms() * 8;
        if (blocks > cap) blocks = cap;
        DEER_KERNEL("ode_discretise_kernel", st, ode_discretise_kernel<<<(unsigned)blocks, ODE_THREADS, sm, st>>>(G, z, t, w.J, w.rhs, B, T, n));
    }
    ScanArgs a{};
    a.J = w.J; a.b = w.rhs; a.y0 = y0; a.y = y; a.yold = nullptr;
    a.B = B; a.T = T; a.n = n; a.reverse = 0;
    a.L = w.scan.L; a.nch = w.scan.nch;
    a.carA = w.scan.carA; a.carB = w.scan.carB; a.starts = w.scan.starts;
    a.st = w.st;
    return run_scan(a, w.scan, flags, st, true, true);
}

size_t deer_multihead_workspace_bytes(const int *strides, int H, int B, int T, int n, int m, int flags)
{
    (void)flags;
    if (!strides || H < 1 || !valid_sizes(B, T, n, m) || !supported(n, m)) return 0;
    for (int h = 0; h < H; ++h)
        if (strides[h] < 1 || (long long)B * strides[h] > 0x7fffffffLL) return 0;
    return carve_mh(nullptr, H, strides, B, T, n, m).bytes;
}

// Heads in order of stride (stable): heads of equal stride read the same dense batch of x, which is then packed once.
static std::vector<int> mh_order(const int *strides, int H)
{
    std::vector<int> order((size_t)H);
    for (int h = 0; h < H; ++h) order[(size_t)h] = h;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return strides[a] < strides[b]; });
    return order;
}

// ---- all heads in one batch: the body, adjoint and contraction kernels take the head as a grid dimension
static bool mh_batched(int n, int H, size_t N, int flags)
{
    return H <= 1024 && N < 0x7fffff00u && body_supported(n, 1, true) &&
           !(flags & (DEER_FLAG_GENERIC | DEER_FLAG_MATERIALIZE | DEER_FLAG_TCGEN05 | DEER_FLAG_EXPIRE_WAITS));
}

// The heads' table on the device; first_edge by the units of `unit` chains of length L (0: none).
static int mh_table(const deer_gru_params *heads, const int *strides, int H, int B, int T, int L, int unit, const MhWs &w, cudaStream_t st)
{
    std::vector<BodyHead> t((size_t)H);
    long long edge = 0, seq = 0;
    for (int h = 0; h < H; ++h) {
        const int s = strides[h], Tp = (T + s - 1) / s;
        t[h] = BodyHead{heads[h].W_i, heads[h].W_h, heads[h].b_i, heads[h].b_h, s, (int)edge, seq};
        if (unit) edge += ((long long)B * s * ((Tp + L - 1) / L) + unit - 1) / unit;
        seq += (long long)B * s;
    }
    if ((size_t)edge > w.groups) return DEER_ERR_WORKSPACE;
    DEER_CHECK_CUDA(cudaMemcpyAsync(w.heads, t.data(), sizeof(BodyHead) * (size_t)H, cudaMemcpyHostToDevice, st), "copy heads");
    return DEER_OK;
}

// u = x W_i^T + b_i of all heads: one contraction [N, m] x [m, H*3n]
static int mh_project(const MhWs &w, const float *x, size_t N, int H, int n, int m, int flags, cudaStream_t st)
{
    DEER_KERNEL("mh_gather_kernel", st, mh_gather_kernel<<<mh_blocks((size_t)H * 3 * n * m), 256, 0, st>>>(w.heads, H, 3 * n, m, w.Wc, w.bc));
    TileGemmArgs a{};
    a.A = x; a.lda = (size_t)m; a.B = w.Wc; a.ldb = (size_t)m; a.bias = w.bc; a.C = w.u;
    a.M = (int)N; a.N = H * 3 * n; a.K = m;
    a.expire = expire_product(flags, 0); a.st = w.st;
    return launch_tile_gemm(TileGemm::MAP, a, 1, st);
}

// The Newton loops of all heads; hs[h].done tells how head h ended (its iterate after hs[h].iters bodies is in y, or, where
// that is odd, in w.yalt).
static int mh_eval_batched(const deer_gru_params *heads, const int *strides, int H, const float *x, const float *y0, int B, int T,
                           float tol, int max_iter, float *y, const MhWs &w, int flags, cudaStream_t st, std::vector<StatusBlock> &hs)
{
    const int n = heads[0].n, m = heads[0].m;
    const size_t N = (size_t)B * T;
    int rc;
    BodyPlan plan{};
    // the two-phase kernel where it is the whole loop in one launch, else the one-phase kernel
    if (!body_plan(&plan, BodyForm::TWO_PHASE, B, T, n, m, true, strides, H) || !plan.whole_loop) {
        plan = BodyPlan{};
        if (!body_plan(&plan, n <= 8 ? BodyForm::LANE : BodyForm::ONE_PHASE, B, T, n, m, true, strides, H)) return DEER_ERR_UNSUPPORTED_N;
    }
    if ((rc = mh_table(heads, strides, H, B, T, plan.L, plan.NC > 0 ? plan.NC : plan.form == BodyForm::LANE ? 32 : 16, w, st)) != DEER_OK) return rc;
    StatusBlock init;
    memset(&init, 0, sizeof(init));
    init.max_iter = max_iter;
    init.tol = tol;
    init.burn = body_first_burn(n, tol);
    const size_t nw = plan.whole_loop ? (size_t)plan.edges * n : 0, nflags = plan.whole_loop ? 0 : (size_t)plan.edges;
    DEER_KERNEL("mh_begin_kernel", st, mh_begin_kernel<<<mh_blocks(nw + nflags + H), 256, 0, st>>>(
                                           w.st, init, H, w.edge_flag, nflags, (unsigned long long *)w.edge, nw, w.words,
                                           plan.whole_loop ? (size_t)4 * H * plan.max_ctas : 0));
    if ((rc = mh_project(w, x, N, H, n, m, flags, st)) != DEER_OK) return rc;
    BodyArgs a{};
    a.heads = w.heads;
    a.u = w.u; a.y0 = y0;
    a.buf[0] = y; a.buf[1] = w.yalt;
    a.B = B; a.T = T; a.n = n; a.m = m; a.H = H; a.L = plan.L;
    a.warm = (flags & DEER_FLAG_WARM_START) ? 1 : 0;
    a.eta = body_eta(n, tol);
    a.burn_cap = plan.burn_cap;
    a.expire = (flags & DEER_FLAG_EXPIRE_BODY_WAITS) != 0;
    a.st = w.st; a.edge = w.edge; a.edge_flag = w.edge_flag; a.words = w.words;
    hs.assign((size_t)H, StatusBlock{});
    for (int group = 4, most = 0;; group = 2) {
        for (int j = 0; j < (plan.whole_loop ? 1 : std::min(group, max_iter - most)); ++j)
            if ((rc = launch_newton_body(a, plan, st)) != DEER_OK) return rc;
        DEER_CHECK_CUDA(cudaMemcpyAsync(hs.data(), w.st, sizeof(StatusBlock) * (size_t)H, cudaMemcpyDeviceToHost, st), "read status");
        DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
        bool all = true;
        most = max_iter;                                 // bodies of the head that is least far
        for (const StatusBlock &h : hs) {
            if (h.flags & FLAG_TIMEOUT) return DEER_ERR_DEVICE_TIMEOUT;
            if (!h.done) { all = false; most = std::min(most, h.iters); }
        }
        if (all) return DEER_OK;
        if (plan.whole_loop) return DEER_ERR_DEVICE_TIMEOUT;
    }
}

// did[h]: the gradients of head h, and its part of dx and dy0, are there (empty: of none).
static int mh_vjp_batched(const deer_gru_params *heads, const int *strides, int H, const float *x, const float *y0, const float *y,
                          const float *gy, int B, int T, const deer_gru_grads *dheads, float *dx, float *dy0, const MhWs &w,
                          int flags, cudaStream_t st, std::vector<char> &did)
{
    const int n = heads[0].n, m = heads[0].m, n3 = 3 * n;
    const size_t N = (size_t)B * T;
    did.clear();
    int rc;
    BodyPlan plan{};
    if (!adjoint_plan(&plan, B, T, n, m, true, strides, H)) return DEER_OK;
    if ((size_t)plan.edges > w.start_groups) return DEER_ERR_WORKSPACE;
    if ((rc = mh_table(heads, strides, H, B, T, plan.L, 16, w, st)) != DEER_OK) return rc;
    std::vector<MhGrad> gr((size_t)H);
    for (int h = 0; h < H; ++h) gr[h] = MhGrad{dheads[h].dW_i, dheads[h].dW_h, dheads[h].db_i, dheads[h].db_h};
    DEER_CHECK_CUDA(cudaMemcpyAsync(w.grads, gr.data(), sizeof(MhGrad) * (size_t)H, cudaMemcpyHostToDevice, st), "copy gradient table");
    StatusBlock init;
    memset(&init, 0, sizeof(init));
    DEER_KERNEL("mh_begin_kernel", st, mh_begin_kernel<<<mh_blocks((size_t)plan.edges + H), 256, 0, st>>>(
                                           w.st, init, H, w.edge_flag, (size_t)plan.edges, nullptr, 0, nullptr, 0));
    if ((rc = mh_project(w, x, N, H, n, m, flags, st)) != DEER_OK) return rc;
    AdjArgs a{};
    a.heads = w.heads;
    a.u = w.u; a.y0 = y0; a.y = y; a.gy = gy;
    a.dGi = w.dGi; a.dGh = w.dGh;
    a.dy0 = dy0 ? w.dy0all : nullptr;
    a.B = B; a.T = T; a.n = n; a.m = m; a.H = H; a.L = plan.L;
    a.eta = ADJ_ETA;
    a.st = w.st; a.edge = w.edge; a.edge_flag = w.edge_flag; a.starts = w.starts;
    a.burn = ADJ_BURN;
    a.burn_cap = 512;                                    // (what comes behind goes head by head)
    for (int k = 0; k < ADJ_TRIES; ++k)
        if ((rc = launch_newton_adjoint(a, plan, st)) != DEER_OK) return rc;
    // dW_i, db_i of all heads: one contraction of dG_i [N, H*3n] with x [N, m]
    TileGemmArgs ga{};
    ga.A = w.dGi; ga.lda = (size_t)H * n3; ga.B = x; ga.ldb = (size_t)m; ga.C = w.partial;
    ga.M = H * n3; ga.N = m; ga.K = (int)N; ga.expire = expire_product(flags, 1); ga.st = w.st;
    const int P = tile_gemm_slices(ga.M, ga.N, ga.K, MH_P_IN);
    if ((rc = launch_tile_gemm(TileGemm::SUMS, ga, P, st)) != DEER_OK) return rc;
    const size_t outs = (size_t)H * n3 * (m + 1);
    DEER_KERNEL("mh_sums_final_kernel", st, mh_sums_final_kernel<<<(unsigned)((outs + 63) / 64), 64 * MH_FINAL, 0, st>>>(w.partial, P, n3, m, H, w.grads, 0, nullptr, nullptr, 0));
    // dW_h, db_h: every head's columns of dG_h with its own of y
    TileGemmArgs gh{};
    gh.A = w.dGh; gh.lda = (size_t)H * n3; gh.B = y; gh.ldb = (size_t)H * n; gh.C = w.partial;
    gh.M = H * n3; gh.N = n; gh.K = (int)N; gh.expire = expire_product(flags, 2); gh.st = w.st;
    gh.heads = w.heads; gh.y0 = y0; gh.T = T; gh.n = n; gh.n3 = n3;
    const int Ph = tile_gemm_slices(gh.M, 1, gh.K, mh_p_hidden(H));
    if ((rc = launch_tile_gemm(TileGemm::SUMS_HEADS, gh, Ph, st)) != DEER_OK) return rc;
    const size_t outs_h = (size_t)H * n3 * (n + 1);
    DEER_KERNEL("mh_sums_final_kernel", st, mh_sums_final_kernel<<<(unsigned)((outs_h + 63) / 64), 64 * MH_FINAL, 0, st>>>(w.partial, Ph, n3, n, H, w.grads, 1, dx ? w.st : nullptr, w.dGi, N));
    if (dx) {
        TileGemmArgs xa{};
        xa.A = w.dGi; xa.lda = (size_t)H * n3; xa.B = w.Wc; xa.ldb = (size_t)m; xa.C = dx;
        xa.M = (int)N; xa.N = m; xa.K = H * n3; xa.expire = expire_product(flags, 3); xa.st = w.st;
        if ((rc = launch_tile_gemm(TileGemm::MAP_T, xa, 1, st)) != DEER_OK) return rc;
    }
    if (dy0) DEER_KERNEL("mh_dy0_sum_kernel", st, mh_dy0_sum_kernel<<<mh_blocks((size_t)B * H * n), 256, 0, st>>>(w.heads, w.dy0all, dy0, B, T, n, H));
    std::vector<StatusBlock> hs((size_t)H);
    DEER_CHECK_CUDA(cudaMemcpyAsync(hs.data(), w.st, sizeof(StatusBlock) * (size_t)H, cudaMemcpyDeviceToHost, st), "read status");
    DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
    if (hs[0].flags & FLAG_TIMEOUT) return DEER_ERR_DEVICE_TIMEOUT;        // (of the dense products)
    for (const StatusBlock &h : hs) did.push_back(h.done == BODY_DONE);    // (a head whose Jacobians hardly decay goes by itself)
    return DEER_OK;
}

int deer_gru_multihead_eval(const deer_gru_params *heads, const int *strides, int H, const float *x, const float *y0,
                            int B, int T, float tol, int max_iter, float *y, int *iters, void *ws, size_t ws_bytes,
                            int flags, void *stream)
{
    int rc = check_mh_args(heads, strides, H, B, T);
    if (rc != DEER_OK) return rc;
    if (!x || !y0 || !y || max_iter < 1 || tol != tol) return DEER_ERR_INVALID_ARG;
    const int n = heads[0].n, m = heads[0].m;
    cudaStream_t st = (cudaStream_t)stream;
    MhWs w = carve_mh(ws, H, strides, B, T, n, m);
    if ((rc = check_ws(ws, ws_bytes, w.bytes)) != DEER_OK) return rc;
    int worst = DEER_OK;
    std::vector<StatusBlock> hs;
    const bool batched = mh_batched(n, H, (size_t)B * T, flags);
    if (batched) {
        if ((rc = mh_eval_batched(heads, strides, H, x, y0, B, T, tol, max_iter, y, w, flags, st, hs)) != DEER_OK) return rc;
        bool odd = false, all = true;
        for (int h = 0; h < H; ++h) {
            odd = odd || (hs[h].iters & 1);
            if (hs[h].done != BODY_DONE) { all = false; continue; }
            float e;
            memcpy(&e, &hs[h].err_last_bits, sizeof(float));
            worst = std::max(worst, eval_status(e, tol));
            if (iters) iters[h] = hs[h].iters;
        }
        if (odd) DEER_KERNEL("mh_select_kernel", st, mh_select_kernel<<<mh_blocks((size_t)B * T * H * n), 256, 0, st>>>(w.st, y, w.yalt, (size_t)B * T, H, n));
        if (all) {
            if (odd) DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
            return worst;
        }
    }
    int packed_stride = 1;                     // stride whose dense batch of x is in w.xs (stride 1: x itself)
    const std::vector<int> order = mh_order(strides, H);
    for (int oi = 0; oi < H; ++oi) {
        const int h = order[(size_t)oi];
        const int s = strides[h], Tp = (T + s - 1) / s, Bs = B * s;
        if (batched && hs[h].done == BODY_DONE) continue;
        const int k0 = batched ? hs[h].iters : 0;      // bodies done before the batched form gave this head up
        if (s != packed_stride) {              // heads of equal stride read the same dense batch of x
            { if ((rc = mh_pack(x, w.xs, B, T, s, Tp, m, m, 0, st)) != DEER_OK) return rc; }
            packed_stride = s;
        }
        const float *xs = s == 1 ? x : w.xs;
        DEER_KERNEL("mh_y0_pack_kernel", st, mh_y0_pack_kernel<<<mh_blocks((size_t)Bs * n), 256, 0, st>>>(y0, w.y0s, B, s, n, H, h));
        if ((flags & DEER_FLAG_WARM_START) || k0 > 0)
            { if ((rc = mh_pack(y, w.ys, B, T, s, Tp, n, H * n, h * n, st)) != DEER_OK) return rc; }
        int it = 0;
        rc = gru_eval_impl(&heads[h], xs, w.y0s, Bs, Tp, tol, max_iter, w.ys, &it, nullptr, nullptr, w.inner, w.inner_bytes,
                           flags, st, nullptr, nullptr, nullptr, nullptr, nullptr, k0);
        if (rc < 0) return rc;
        if (iters) iters[h] = it;
        if (rc > worst) worst = rc;
        { if ((rc = mh_unpack(w.ys, y, B, T, s, Tp, n, H * n, h * n, 0, st)) != DEER_OK) return rc; }
    }
    DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
    return worst;
}

int deer_gru_multihead_vjp(const deer_gru_params *heads, const int *strides, int H, const float *x, const float *y0,
                           const float *y, const float *gy, int B, int T, const deer_gru_grads *dheads, float *dx,
                           float *dy0, void *ws, size_t ws_bytes, int flags, void *stream)
{
    int rc = check_mh_args(heads, strides, H, B, T);
    if (rc != DEER_OK) return rc;
    if (!x || !y0 || !y || !gy || !dheads) return DEER_ERR_INVALID_ARG;
    for (int h = 0; h < H; ++h)
        if (!dheads[h].dW_i || !dheads[h].dW_h || !dheads[h].db_i || !dheads[h].db_h) return DEER_ERR_INVALID_ARG;
    const int n = heads[0].n, m = heads[0].m;
    cudaStream_t st = (cudaStream_t)stream;
    MhWs w = carve_mh(ws, H, strides, B, T, n, m);
    if ((rc = check_ws(ws, ws_bytes, w.bytes)) != DEER_OK) return rc;
    std::vector<char> did;
    if (mh_batched(n, H, (size_t)B * T, flags) &&
        (rc = mh_vjp_batched(heads, strides, H, x, y0, y, gy, B, T, dheads, dx, dy0, w, flags, st, did)) != DEER_OK) return rc;
    const bool batched = !did.empty();
    unsigned timeout_flags = 0;
    int packed_stride = 1;                     // (stride 1: x itself)
    const std::vector<int> order = mh_order(strides, H);
    for (int oi = 0; oi < H; ++oi) {
        const int h = order[(size_t)oi];
        const int s = strides[h], Tp = (T + s - 1) / s, Bs = B * s;
        if (batched && did[(size_t)h]) continue;
        if (s != packed_stride) {
            { if ((rc = mh_pack(x, w.xs, B, T, s, Tp, m, m, 0, st)) != DEER_OK) return rc; }
            packed_stride = s;
        }
        const float *xs = s == 1 ? x : w.xs;
        DEER_KERNEL("mh_y0_pack_kernel", st, mh_y0_pack_kernel<<<mh_blocks((size_t)Bs * n), 256, 0, st>>>(y0, w.y0s, B, s, n, H, h));
        { if ((rc = mh_pack(y, w.ys, B, T, s, Tp, n, H * n, h * n, st)) != DEER_OK) return rc; }
        { if ((rc = mh_pack(gy, w.gys, B, T, s, Tp, n, H * n, h * n, st)) != DEER_OK) return rc; }
        rc = gru_vjp_impl(&heads[h], xs, w.y0s, w.ys, w.gys, Bs, Tp, &dheads[h], dx ? w.dxs : nullptr, dy0 ? w.dy0s : nullptr,
                          w.inner, w.inner_bytes, flags, st);
        if (rc != DEER_OK) return rc;
        if (dx)     // the heads' input gradients add up, head by head in a fixed order (that of the strides; behind those of a batch)
            { if ((rc = mh_unpack(w.dxs, dx, B, T, s, Tp, m, m, 0, batched || oi > 0, st)) != DEER_OK) return rc; }
        if (dy0)
            DEER_KERNEL("mh_dy0_reduce_kernel", st, mh_dy0_reduce_kernel<<<mh_blocks((size_t)B * n), 256, 0, st>>>(w.dy0s, dy0, B, s, n, H, h));
        // the inner gradient calls share one status block: keep every head's flags
        unsigned f = 0;
        DEER_CHECK_CUDA(cudaMemcpyAsync(&f, &reinterpret_cast<const StatusBlock *>(w.inner)->flags, sizeof(unsigned),
                                        cudaMemcpyDeviceToHost, st), "read status");
        DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
        timeout_flags |= f;
    }
    return (timeout_flags & FLAG_TIMEOUT) ? DEER_ERR_DEVICE_TIMEOUT : DEER_OK;
}

int deer_linrec_scan_noalloc(const float *J, const float *b, const float *y0, int B, int T, int n,
                             int reverse, float *y, void *stream)
{
    if (!J || !b || !y || B <= 0 || T <= 0 || n <= 0) return DEER_ERR_INVALID_ARG;
    if (!supported(n, 1)) return DEER_ERR_UNSUPPORTED_N;
    if (!valid_sizes(B, T, n, 1)) return DEER_ERR_INVALID_ARG;
    const size_t need = carve_scan_only(nullptr, B, T, n).scan.bytes_without;
    if (need > sizeof(g_noalloc_scratch)) {
        snprintf(t_err, sizeof(t_err),
                 "deer_linrec_scan_noalloc: B=%d T=%d n=%d needs %zu bytes of scratch, the built-in array holds %zu",
                 B, T, n, need, sizeof(g_noalloc_scratch));
        return DEER_ERR_WORKSPACE;
    }
    void *scratch = nullptr;
    int rc = noalloc_scratch_for_current_device(&scratch);
    if (rc != DEER_OK) return rc;
    // linrec_scan_impl clears what has to start at zero (status block, tile flags, entering-state
    // words, counters) with stream-ordered memsets on every call; nothing else is read before written
    return linrec_scan_impl(J, b, y0, B, T, n, reverse, y, scratch, sizeof(g_noalloc_scratch), 0,
                            (cudaStream_t)stream);
}

static int status_from_block(const void *block, cudaStream_t st)
{
    StatusBlock hs;
    DEER_CHECK_CUDA(cudaMemcpyAsync(&hs, block, 32, cudaMemcpyDeviceToHost, st), "read status");
    DEER_CHECK_CUDA(cudaStreamSynchronize(st), "sync");
    return (hs.flags & FLAG_TIMEOUT) ? DEER_ERR_DEVICE_TIMEOUT : DEER_OK;
}

int deer_workspace_status(const void *ws, void *stream)
{
    if (!ws || ((uintptr_t)ws & 255) != 0) return DEER_ERR_WORKSPACE;
    return status_from_block(ws, (cudaStream_t)stream);
}

int deer_noalloc_status(void *stream)
{
    void *scratch = nullptr;
    int rc = noalloc_scratch_for_current_device(&scratch);
    if (rc != DEER_OK) return rc;
    return status_from_block(scratch, (cudaStream_t)stream);
}

int deer_scan_geometry(int B, int T, int n, int flags, int *out)
{
    if (!out || B <= 0 || T <= 0 || n <= 0) return DEER_ERR_INVALID_ARG;
    if (!supported(n, 1)) return DEER_ERR_UNSUPPORTED_N;
    if (!valid_sizes(B, T, n, 1)) return DEER_ERR_INVALID_ARG;
    const bool umma = (flags & DEER_FLAG_TCGEN05) != 0;
    int sw = 0;
    const int L1 = onepass_tile_len(n, B, T, &sw);
    const bool single = L1 > 0 && !(flags & DEER_FLAG_GENERIC) && B <= single_pass_max_batch(n, umma);
    if (single) {
        int res_warps = 0, max_seq = 0, res_cap = 8;
        switch (n) {
        case 1: case 2: case 4: res_warps = n == 4 ? OnePass<4>::WARPS : OnePass<1>::WARPS; max_seq = OnePass<1>::MAX_SEQ_PER_WARP; break;
        case 8: res_warps = Warp8::RES_WARPS; max_seq = OnePass<8>::MAX_SEQ_PER_WARP; break;
        case 16: case 32: res_warps = big_res_warps(B); max_seq = WarpN<16>::MAX_SEQ_PER_WARP; break;
        default: res_warps = umma ? Umma64::RES_WARPS : res_warps64(B); max_seq = Cta64::MAX_SEQ_PER_WARP; res_cap = umma ? 8 : 16; break;
        }
        out[0] = 1; out[1] = L1; out[2] = sw; out[3] = (T + L1 - 1) / L1;
        out[4] = resolver_ctas(B, res_warps, max_seq, res_cap);
    } else {
        const int L = gen_chunk_len(T);
        out[0] = 0; out[1] = L; out[2] = 0; out[3] = (T + L - 1) / L; out[4] = 0;
    }
    out[5] = num_sms();
    return DEER_OK;
}

int deer_gru_cell_jac(const deer_gru_params *p, const float *x, const float *y0, const float *y, int B, int T,
                      float *J, float *rhs, void *ws, size_t ws_bytes, int flags, void *stream)
{
    if (!p || !x || !y0 || !y || !J || !rhs || !p->W_i || !p->W_h || !p->b_i || !p->b_h) return DEER_ERR_INVALID_ARG;
    if (B <= 0 || T <= 0 || p->n <= 0 || p->m <= 0) return DEER_ERR_INVALID_ARG;
    if (!supported(p->n, p->m)) return DEER_ERR_UNSUPPORTED_N;
    if (!valid_sizes(B, T, p->n, p->m)) return DEER_ERR_INVALID_ARG;
    const int n = p->n, m = p->m;
    const bool coef = (flags & DEER_FLAG_COEF_ROWS) != 0;
    if (coef && !(n == 16 || n == 32 || n == 64)) return DEER_ERR_UNSUPPORTED_N;
    if (coef && (flags & DEER_FLAG_GENERIC)) return DEER_ERR_INVALID_ARG;
    if (coef && ((((uintptr_t)y | (uintptr_t)y0 | (uintptr_t)J | (uintptr_t)p->W_h) & 15) != 0)) return DEER_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    EvalWs w = carve_eval(ws, B, T, n, m);
    int rc = check_ws(ws, ws_bytes, w.bytes);
    if (rc != DEER_OK) return rc;
    const bool generic = (flags & DEER_FLAG_GENERIC) != 0;
    const bool fused_proj = !generic && cell_projects(n, m) && ((((uintptr_t)y | (uintptr_t)y0 | (uintptr_t)J) & 15) == 0);
    if (!fused_proj && (rc = run_proj(p, x, w.u, (size_t)B * T, st)) != DEER_OK) return rc;
    CellArgs c{p->W_h, p->b_h, fused_proj ? nullptr : w.u, x, p->W_i, p->b_i, m, y, y0, J, rhs, B, T, n, nullptr, coef ? 1 : 0};
    return run_cell(c, st, generic);
}

const char *deer_status_string(int s)
{
    switch (s) {
    case DEER_OK: return "ok";
    case DEER_NOT_CONVERGED: return "not converged within max_iter";
    case DEER_NONFINITE: return "non-finite values in the iterate";
    case DEER_ERR_INVALID_ARG: return "invalid argument";
    case DEER_ERR_UNSUPPORTED_N: return "unsupported hidden or input size";
    case DEER_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
    case DEER_ERR_CUDA: return "CUDA runtime error";
    case DEER_ERR_DEVICE_TIMEOUT: return "bounded device-side wait expired";
    default: return "unknown status";
    }
}

const char *deer_last_error(void) { return t_err; }

long long deer_launch_count(void) { return g_launches.load(); }

void deer_profile_enable(int on)
{
    g_prof_on.store(on != 0);
}

size_t deer_profile_read(char *buf, size_t cap)
{
    std::lock_guard<std::mutex> lk(g_prof_mu);
    std::map<std::string, std::pair<long, double>> acc;
    std::vector<std::string> order;
    for (auto &r : g_prof) {
        float ms = 0.0f;
        cudaEventSynchronize(r.e1);
        cudaEventElapsedTime(&ms, r.e0, r.e1);
        cudaEventDestroy(r.e0);
        cudaEventDestroy(r.e1);
        if (!acc.count(r.name)) order.push_back(r.name);
        acc[r.name].first += 1;
        acc[r.name].second += ms;
    }
    g_prof.clear();
    std::string out;
    char line[160];
    for (auto &k : order) {
        snprintf(line, sizeof(line), "%s %ld %.6f\n", k.c_str(), acc[k].first, acc[k].second);
        out += line;
    }
    if (buf && cap) {
        size_t c = out.size() < cap - 1 ? out.size() : cap - 1;
        memcpy(buf, out.data(), c);
        buf[c] = 0;
    }
    return out.size();
}

}  // extern "C"
