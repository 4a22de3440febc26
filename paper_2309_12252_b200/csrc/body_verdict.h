// The decision at the end of a one-launch Newton body: plain arithmetic, for device and host alike.
#pragma once
#include <math.h>
#ifdef __CUDACC__
#define DEER_HD __host__ __device__ __forceinline__
#else
#include <algorithm>
#define DEER_HD inline
#endif

namespace deer {

#ifndef __CUDACC__
using std::max;
using std::min;
#endif

// StatusBlock::done: the loop ended / this form gives up / a bounded wait ran out, nothing that was computed counts / the tiles
// take the inputs in units of their own (tile_units_kernel) / a value is beyond f16's range, or not finite at all: what runs
// without such an operand tells, and no burn-in is told
constexpr int BODY_DONE = 1, BODY_FALL_BACK = 2, BODY_TIMED_OUT = 3, BODY_UNITS = 4, BODY_BEYOND = 5;

constexpr int BODY_BURN_MIN = 8; // shortest burn-in that is tried
constexpr float BODY_ROUNDING = 2.4e-7f;         // two roundings of a state below one in size

DEER_HD bool newton_loop_ends(float e, float tol, int k, int max_iter)
{
    return !(e > tol) || !(e <= 3.402823466e38f) || k + 1 >= max_iter;
}

DEER_HD float verdict_log(float x)
{
#ifdef __CUDA_ARCH__
    return __logf(x);
#else
    return logf(x);
#endif
}

// What becomes of a body whose update is e and whose largest boundary mismatch is mis, and the burn-in of the next one.
//
// Where the loop runs to a tolerance, a body whose boundaries are good to a thousandth of its update is a good quasi-Newton
// step: it counts.  Far from the solution more than that is lost in Newton's own quadratic error (updates of 1.7, 0.8, 0.05
// are usual): a twentieth of the update times the update is then good enough.  (Slowly varying inputs, n = 32, B = 16,
// T = 2e4: two of six bodies were run again for it.)
//
// The carried error is about e * rho^burn, so a body shows the rate at which its cell forgets.  What proves too short is raised
// to what that rate calls for.  Where chains are short, so that a body's time goes with its burn-in (`adapt`), the next body gets
// the steps that its own accuracy calls for and no more: a quarter of eta of its update (or of the tolerance, whichever is
// more), or of what counts far from the solution, its update being expected between 0.1 and 2 times this one's square (0.06 ...
// 0.43 were seen).  Behind a zero guess the rate is not yet the solution's -- slowly varying inputs lost up to half of it from the
// first body to the second -- so the second one gets a third more.  (Steps per body of a fixed burn-in raised on need, and so:
// n = 24, B = 5, T = 4,001, random walks 30 53 53 53 -> 24 37 37 42; n = m = 32, B = 16, T = 1e5, white noise 24 24 24 24 -> 16 22
// 19 15, 1370 -> 1292 us.)
//
// `rounding`: what the mismatch is off by where the update is the difference of two rounded states below one in size.  A carried
// error of that size looks the same, so it passes only where it is small beside the tolerance: up to 2.5e-3 of that, as much as a
// good quasi-Newton step leaves anyway.  Below a tolerance of 1e-4 the other kernels finish what rounding makes undecidable here.
struct BodyVerdict { bool counts; int done, burn, need; };   // need: the burn-in for eta itself (0: this body does not tell)
DEER_HD BodyVerdict body_verdict(float e, float mis, float eta, int burn, int burn_cap, int T, float tol, int iters, int max_iter, bool adapt, float rounding)
{
    BodyVerdict v{true, 0, burn, 0};
    if (e <= 3.402823466e38f) {                          // (a NaN or Inf ends the loop)
        const bool to_tol = tol > 0.0f;
        const float scale = fmaxf(e, to_tol ? tol : 0.0f), thr = eta * scale, slack = to_tol ? fminf(rounding, 2.5e-3f * tol) : 0.0f;
        const float near = fmaxf(eta, 1e-3f) * scale, most = to_tol ? fmaxf(fmaxf(near, slack), 0.05f * fminf(e, 1.0f) * e) : thr;
        const int never = 1 << 20, whole = max(T, burn);                 // (a burn-in of the whole sequence is exact)
        const float ratio = mis / e;
        // steps that take an error down to `part` of itself (what is below 1e-7 of the update is rounding)
        auto steps = [&](float part) { return ratio < 0.7f ? (int)((float)burn * verdict_log(part) / verdict_log(fmaxf(ratio, 1e-7f))) : never; };
        if (!(mis <= 2.0f * rounding)) v.need = min(steps(0.5f * eta), whole);
        if (!(mis <= fmaxf(thr, slack))) {
            auto raised = [&](int n) { return min(max(n < never ? n + n / 10 + 4 : n, burn + 8), whole); };
            const int wn = raised(steps(0.5f * thr / e));
            if (!(mis <= most)) {
                v.counts = false;
                v.burn = wn;
                if (adapt && to_tol) {
                    // (no kernel is given more than burn_cap: the two-phase form's shared memory holds no more positions)
                    v.burn = min(min(wn, max(burn + 8, steps(0.25f * most / e) * 5 / 4)), burn_cap);
                    if (v.burn <= burn || raised(steps(0.5f * near / e)) > burn_cap) {               // (the bodies behind it have to be that good)
                        v.done = BODY_FALL_BACK;
                        v.burn = wn;                     // (what eta would need is what is told: a gradient's first burn-in comes from it)
                    }
                } else if (wn > burn_cap) {
                    v.done = BODY_FALL_BACK;
                }
                return v;
            }
            v.burn = min(wn, burn_cap);
            if (wn > burn_cap && !(mis <= fmaxf(near, slack))) v.done = BODY_FALL_BACK;         // (it would not do for the next one)
        }
        if (adapt && to_tol && e > tol && !v.done) {
            const float lo = 0.1f * e * e, hi = fminf(e, 2.0f * e * e);
            const float part = 0.25f * fmaxf(eta * fmaxf(1.0f, tol / hi), 0.05f * fminf(lo, 1.0f));
            int wn = steps(part) + 1;
            if (iters == 0) wn += wn / 3;
            v.burn = min(min(max(wn, BODY_BURN_MIN), burn_cap), whole);
        }
    }
    if (newton_loop_ends(e, tol, iters, max_iter)) v.done = BODY_DONE;
    return v;
}

}  // namespace deer
