// One Newton body of an evaluation as ONE launch (see newton_body.cuh): host-side interface.
#pragma once
#include "common.cuh"

namespace deer {

// One cell (head) of a launch: its parameters and the stride of its time axis.
struct BodyHead {
    const float *W_i, *W_h, *b_i, *b_h;
    int stride;              // a head of stride s runs s interleaved sequences per batch entry
    int first_edge;          // offset of the head's chain groups in the edge buffers
    long long first_seq;     // sequences of the heads before this one (adjoint: rows of dy0)
};

struct BodyArgs {
    BodyHead h0;             // the only head when `heads` is null
    const BodyHead *heads;   // device array [H]
    const float *x;          // [B,T,m]      contracted in the kernel (u == nullptr)
    const float *u;          // [B,T,H,3n]   or: x W_i^T + b_i of every head
    const float *y0;         // [B,H,n]
    float *buf[2];           // [B,T,H,n]    iterate k in buf[k & 1]
    int B, T, n, m, H;
    int L;                   // positions a chain owns
    int warm;                // buf[0] holds the guess (0: the guess is zero and buf[0] is not read)
    float eta;               // largest boundary mismatch, as a part of max(err, tol), that is accepted
    int burn_cap;            // longest burn-in that is tried (BodyPlan)
    int expire;              // test aid: every bounded wait runs out (DEER_FLAG_EXPIRE_BODY_WAITS)
    int polled;              // the host reads the result record while the stream runs
    int units;               // tiles: x comes from launch_tile_units
    int adapt;               // chains so short that a body's burn-in is its time: no longer than its own accuracy calls for
    StatusBlock *st;         // [H]
    float *edge;             // [groups][2][n]  states either side of a boundary between two warps
    unsigned *edge_flag;     // [groups]        arrivals at it (left cleared)
    float *starts;           // [chains][n]     tile kernel: update that each chain assumed at its first own position
    unsigned long long *words;   // [H][2][CTAs][2]  maxima exchanged at the end of a body (whole-loop launches)
};

// The adjoint solve of the gradient as one launch (newton_adjoint.cuh).
struct AdjArgs {
    BodyHead h0;
    const BodyHead *heads;
    const float *x, *u, *y0; // as in BodyArgs
    const float *y, *gy;     // [B,T,H,n] trajectory, dL/dy
    const float *gy_seq;     // tiles, or nullptr: [B,n] dL/dy where it is the same at every step of a sequence (gy is not read)
    float *lam;              // [B,T,H,n] out: lambda; or nullptr:
    float *dGi, *dGh;        // [B,T,H,3n] out: gradients w.r.t. the input-side and hidden-side pre-activations
    int packed;              // one head: dGi receives rows [4n] = (r, z, n hidden, n input) and dGh nothing
    float *dy0;              // or nullptr; row b * H + head (dy0_by_head), else first_seq + sequence
    int dy0_by_head;
    int B, T, n, m, H, L;
    int burn, burn_cap;      // burn-in of the first try; longest that another one is worth
    float eta;               // largest boundary mismatch that is accepted, as a part of max|lambda| (and see ADJ_LOCAL)
    int expire;              // as in BodyArgs
    StatusBlock *st;         // [H]; done = 1 where the launch has done the work (it returns at once where it is set)
    float *edge;             // [boundaries][ADJ_EDGE(n)]  end state of the chain before, start state and scale of the one behind
    unsigned *edge_flag;
    float *starts;           // [groups][16][n + 4 of the padded size], n > 48 only (adjoint_starts)
};

__host__ __device__ constexpr int ADJ_EDGE(int n) { return 2 * n + 1; }

// The kernels of one padded state size (newton_kernels.cu).
struct BodyKernels {
    void (*one)(BodyArgs);                     // one-phase (newton_body.cuh); n > 8 only
    void (*seg)(BodyArgs, int, int);           // two-phase (newton_segment.cuh)
    void (*(*adj)(int m))(AdjArgs);            // adjoint, one-phase (newton_adjoint.cuh); m: channels contracted in the kernel
    void (*(*tile)(int m))(BodyArgs);          // 128 chains per tcgen05 tile (newton_tile.cuh); n = 32, 64 only
    size_t (*tile_smem)(int m);
    void (*tile_units)(const float *x, float *xs, size_t count, int m, const float *W_h, const float *W_i);
    int tile_threads, tile_chains;
    void (*(*adj_tile)(int m))(AdjArgs);
    size_t (*adj_tile_smem)(int m);
    int one_warps, seg_warps, nc_max;
    size_t slot_bytes;
    size_t (*one_smem)(int kx), (*seg_fixed)(int kx), (*adj_smem)(int kx);
};

constexpr int BODY_L_MIN = 3;    // chains are at least this long
constexpr int CHAIN_L_MIN = 4;   // ... those of every form but the two-phase one: what boundaries and start states are sized by

// The forms of a body.
enum class BodyForm { TWO_PHASE, TILE, LANE, ONE_PHASE };

// How a body is launched.
struct BodyPlan {
    BodyForm form;
    int NC;                  // > 0: the two-phase kernel, chains per CTA (newton_segment.cuh); 0: the one-phase kernel
    int L;                   // positions per chain
    int warps;               // warps per CTA
    int max_ctas;            // grid.x: CTAs of the head that needs most
    int burn_cap;            // longest burn-in the launch can hold or is worth trying
    bool whole_loop;         // the whole Newton loop is one (cooperative) launch
    float waves;             // CTAs of the launch / CTAs that the GPU holds
    float share;             // positions per chain if every chain that the GPU holds at a time had the same (one-phase, tile, lane)
    long long edges;         // boundaries between warps (one-phase) or CTAs (two-phase) of all heads at most
    size_t smem;
};

// The whole gradient of a small cell in one launch (rows_adjoint.cuh): n, m in {1, 2, 4, 8}; the launch writes
// plan.max_ctas slices of the parameter gradients.
struct RowsAdjOut;
bool rows_adjoint_plan(BodyPlan *p, int B, int T, int n, int m, int max_ctas);
int launch_rows_adjoint(const AdjArgs &a, const BodyPlan &p, float *partial_i, float *partial_h, float *dx, cudaStream_t st);
void (*rows_adjoint_of(int n, int m))(AdjArgs, RowsAdjOut);

// A thread per chain (newton_lane.cuh): n up to 8; inputs of up to 8 channels contracted in the kernel, else projected.
struct LaneKernel { void (*kern)(BodyArgs); size_t smem; int W; };
LaneKernel lane_kernel(int n, int m, bool have_u);

// Does the kernel take these sizes?
bool body_supported(int n, int m, bool have_u);
// Chain length and launch shape of a form; strides == nullptr: one head of stride 1.  False when the form does not take these
// sizes.
bool body_plan(BodyPlan *p, BodyForm form, int B, int T, int n, int m, bool have_u, const int *strides, int H);
// Does the form the plan stands for suit the problem, or are the kernels that multiply the Jacobians out faster?
bool body_suits(const BodyPlan &p, int n);
// Burn-in that a cell as initialised needs for the accuracy asked of the boundaries, that accuracy, and the burn-in of the first
// body behind a zero guess.
int body_first_burn(int n, float tol);
int body_start_burn(int n, float tol, bool adapt);
float body_eta(int n, float tol);
int launch_newton_body(const BodyArgs &a, const BodyPlan &p, cudaStream_t st);
// xs [B,T,m]: x in the units of the tiles' operands, for BodyArgs::units.
int launch_tile_units(const BodyArgs &a, float *xs, cudaStream_t st);

bool adjoint_supported(int n, int m, bool have_u);
bool adjoint_plan(BodyPlan *p, int B, int T, int n, int m, bool have_u, const int *strides, int H);
// floats of AdjArgs::starts per chain group (0: not used)
size_t adjoint_starts(int n);
// Longest burn-in for which a launch of chains of L beats the kernels that multiply the Jacobians out.
int adjoint_burn_cap(int n, int m, long long positions, int L);
int launch_newton_adjoint(const AdjArgs &a, const BodyPlan &p, cudaStream_t st);
// The same with 128 chains per tcgen05 tile (adjoint_tile.cuh): n = 64; AdjArgs::dGi receives packed rows [4n].
bool adjoint_tile_plan(BodyPlan *p, int B, int T, int n, int m);
int launch_adjoint_tile(const AdjArgs &a, const BodyPlan &p, cudaStream_t st);
// Launches of a gradient (the second with the burn-in that the first one found), the first one's burn-in, and the accuracy
// asked of the boundaries (a one-shot solve: fp32 level).
constexpr int ADJ_TRIES = 2, ADJ_BURN = 44;
constexpr float ADJ_ETA = 4e-6f;

}  // namespace deer
