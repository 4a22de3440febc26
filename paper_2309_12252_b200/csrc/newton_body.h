// One Newton body of an evaluation as ONE launch (see newton_body.cuh): host-side interface.
#pragma once
#include "common.cuh"

namespace deer {

// One cell (head) of a launch: its parameters and the stride of its time axis.
struct BodyHead {
    const float *W_i, *W_h, *b_i, *b_h;
    int stride;              // a head of stride s runs s interleaved sequences per batch entry
    int first_edge;          // offset of the head's chain groups in the edge buffers
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
    StatusBlock *st;         // [H]
    float *edge;             // [groups][2][n]  states either side of a boundary between two warps
    unsigned *edge_flag;     // [groups]        arrivals at it (left cleared)
    unsigned long long *words;   // [H][2][CTAs][2]  maxima exchanged at the end of a body (whole-loop launches)
};

constexpr int BODY_DONE = 1, BODY_FALL_BACK = 2;       // StatusBlock::done: the loop ended / this form gives up

// The kernels of one padded state size (newton_kernels.cu).
struct BodyKernels {
    void (*one)(BodyArgs);                     // one-phase (newton_body.cuh)
    void (*seg)(BodyArgs, int, int);           // two-phase (newton_segment.cuh)
    int one_warps, seg_warps, nc_max;
    size_t slot_bytes;
    size_t (*one_smem)(int kx), (*seg_fixed)(int kx);
};

constexpr int BODY_L_MIN = 3;    // chains are at least this long

// How a body is launched.
struct BodyPlan {
    int NC;                  // > 0: the two-phase kernel, chains per CTA (newton_segment.cuh); 0: the one-phase kernel
    int L;                   // positions per chain
    int warps;               // warps per CTA
    int max_ctas;            // grid.x: CTAs of the head that needs most
    int burn_cap;            // longest burn-in the launch can hold or is worth trying
    bool whole_loop;         // the whole Newton loop is one (cooperative) launch
    float waves;             // CTAs of the launch / CTAs that the GPU holds
    long long edges;         // boundaries between warps (one-phase) or CTAs (two-phase) of all heads at most
    size_t smem;
};

// Does the kernel take these sizes?
bool body_supported(int n, int m, bool have_u);
// Chain length and launch shape; strides == nullptr: one head of stride 1.  two_phase: the form to plan for; returns
// false when it does not take these sizes.
bool body_plan(BodyPlan *p, bool two_phase, int B, int T, int n, int m, bool have_u, const int *strides, int H);
// Does the form the plan stands for suit the problem, or are the kernels that multiply the Jacobians out faster?
bool body_suits(const BodyPlan &p, int n);
// Burn-in a call starts with, and the accuracy asked of the boundaries.
int body_first_burn(int n, float tol);
float body_eta(int n, float tol);
int launch_newton_body(const BodyArgs &a, const BodyPlan &p, cudaStream_t st);

}  // namespace deer
