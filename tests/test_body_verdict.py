"""The decision at the end of a one-launch Newton body (csrc/body_verdict.h), as host code."""
import ctypes
import math
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2309_12252_b200", "csrc")

HARNESS = r'''
#include "body_verdict.h"
using namespace deer;
extern "C" void verdict(float e, float mis, float eta, int burn, int cap, int T, float tol, int iters, int adapt, float rounding, int *out)
{
    const BodyVerdict v = body_verdict(e, mis, eta, burn, cap, T, tol, iters, 100, adapt != 0, rounding);
    out[0] = v.counts; out[1] = v.done; out[2] = v.burn; out[3] = v.need;
}
// Bodies whose boundaries forget by `rho` a step, over updates, burn-ins, limits and accuracies: those that end nothing and would
// have the next body run a burn-in beyond the limit (over), or the same body again with no more of it (stuck).
extern "C" void sweep(long long *looked_at, long long *over, long long *stuck)
{
    *looked_at = *over = *stuck = 0;
    const float etas[] = {1e-3f, 1e-4f, 4e-6f}, tols[] = {1e-4f, 1e-6f, 1e-2f, -1.0f};
    for (float eta : etas) for (float tol : tols) for (int cap : {30, 96, 97, 128, 224, 320, 512}) for (int T : {50, 128, 100000})
    for (int adapt = 0; adapt < 2; ++adapt) for (int iters = 0; iters < 3; ++iters) for (float rounding : {0.0f, BODY_ROUNDING})
    for (int burn = 8; burn <= cap && burn < T; burn += 1 + burn / 8)          // (from T on every chain starts at its sequence's first step)
    for (float e = 1e-6f; e < 1e3f; e *= 3.0f) for (float rho = 0.4f; rho < 1.02f; rho += 0.015f) {
        const BodyVerdict v = body_verdict(e, e * powf(rho, (float)burn), eta, burn, cap, T, tol, iters, 100, adapt != 0, rounding);
        ++*looked_at;
        if (!v.done && v.burn > cap) ++*over;
        if (!v.done && !v.counts && v.burn <= burn) ++*stuck;
    }
}
'''


@pytest.fixture(scope="module")
def V(tmp_path_factory):
    d = tmp_path_factory.mktemp("verdict")
    src, lib = str(d / "harness.cpp"), str(d / "harness.so")
    with open(src, "w") as f:
        f.write(HARNESS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", lib], check=True)
    return ctypes.CDLL(lib)


def test_no_body_is_given_a_burn_in_beyond_the_limit(V):
    """The two-phase kernel's shared memory holds the limit's positions and no more."""
    looked_at, over, stuck = (ctypes.c_longlong() for _ in range(3))
    V.sweep(ctypes.byref(looked_at), ctypes.byref(over), ctypes.byref(stuck))
    assert looked_at.value > 1_000_000
    assert over.value == 0 and stuck.value == 0, (over.value, stuck.value)


def verdict(V, e, mis, eta, burn, cap, T, tol, iters, adapt, rounding=0.0):
    out = (ctypes.c_int * 4)()
    f = ctypes.c_float
    V.verdict(f(e), f(mis), f(eta), burn, cap, T, f(tol), iters, int(adapt), f(rounding), out)
    return dict(counts=out[0], done=out[1], burn=out[2], need=out[3])


FALL_BACK = 2


@pytest.mark.parametrize("rho", [0.93, 0.95, 0.97])
@pytest.mark.parametrize("eta", [1e-3, 1e-4])
def test_a_form_that_gives_up_tells_what_its_boundaries_would_need(V, rho, eta):
    """Whatever the next body would have been given: the steps after which half of eta of the update is left."""
    e, burn = 1e-2, 30
    told = [verdict(V, e, e * rho ** burn, eta, burn, 64, 100000, 1e-4, 1, adapt) for adapt in (False, True)]
    assert all(v["done"] == FALL_BACK and not v["counts"] for v in told), told
    assert told[0]["burn"] == told[1]["burn"] >= math.log(0.5 * eta) / math.log(rho), told


@pytest.mark.parametrize("eta", [1e-3, 1e-4])
@pytest.mark.parametrize("tol", [1e-3, 1e-4, 1e-5, 1e-6, 1e-7, 1e-9])
@pytest.mark.parametrize("rounding", [0.0, 2.4e-7])
def test_an_evaluation_does_not_end_on_a_boundary_that_is_off_by_more_than_its_tolerance_allows(V, eta, tol, rounding):
    """The last body's boundaries are good to 2.5e-3 of the tolerance, whatever its states are rounded to; at 1e-4 rounding is no
    reason to run it again."""
    for mis in (1e-12, 1e-10, 3e-9, 6e-8, 1.2e-7, 2.4e-7, 1e-6, 1e-5):
        v = verdict(V, 0.5 * tol, mis, eta, 30, 512, 100000, tol, 3, False, rounding)
        if v["counts"]:
            assert mis <= 2.5e-3 * tol * (1 + 1e-6), mis
        elif rounding and mis <= 2.4e-7:
            assert tol < 1e-4, mis


@pytest.mark.parametrize("eta", [1e-3, 1e-4])
def test_the_next_burn_in_follows_the_decay(V, eta):
    """Short chains: the steps that take the next update's error, of about the square of this one, down to a quarter of what it is
    asked for, at the rate that this body showed, and a third more behind a zero guess.  Others keep theirs."""
    e, burn = 0.1, 24
    for iters in (0, 2):
        got = []
        for rho in (0.52, 0.57, 0.62, 0.67, 0.72):            # (0.52^24: what is below 1e-7 of an update is rounding)
            v = verdict(V, e, e * rho ** burn, eta, burn, 512, 100000, 1e-4, iters, True)
            assert v["counts"] and not v["done"]
            want = math.log(0.25 * max(eta, 0.05 * 0.1 * e * e)) / math.log(rho) * (4 / 3 if iters == 0 else 1)
            assert abs(v["burn"] - max(8, want)) <= 2, (rho, v)
            got.append(v["burn"])
            assert verdict(V, e, e * rho ** burn, eta, burn, 512, 100000, 1e-4, iters, False)["burn"] == burn or rho ** burn > eta
        assert got == sorted(got) and got[-1] >= 1.8 * got[0]
        assert verdict(V, e, e * 0.72 ** burn, eta, burn, burn, 100000, 1e-4, iters, True)["burn"] == burn
