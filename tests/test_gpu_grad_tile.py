"""The one-pass contractions of a gradient: where its tiles, padded columns, sequence starts and flushes can go wrong."""
import numpy as np
import pytest
import torch

import oracle
from paper_2309_12252_b200 import binding as bd
from paper_2309_12252_b200 import synth

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# runs of 64 positions: fewer than one, one more than one, sequences shorter than a run, a last run that is nearly empty, several
# flushes; state sizes on and off the padded 32 and 64, inputs on and off multiples of 4 and 16, up to the most that it takes
@pytest.mark.parametrize("n,m,B,T,scale", [
    (32, 32, 1, 1, 1.0), (64, 64, 1, 65, 1.0), (32, 5, 70, 7, 1.0), (16, 1, 3, 64, 1e-30), (20, 64, 3, 400, 1.0), (24, 10, 5, 801, 1e-30),
    (32, 33, 2, 999, 1e20), (32, 48, 1, 128, 1.0), (48, 17, 2, 450, 1.0), (60, 63, 3, 301, 1e-30), (64, 6, 5, 1501, 1.0),
    (36, 40, 1, 2000, 1.0), (32, 32, 16, 40001, 1.0), (64, 64, 8, 20001, 1.0),
])
def test_gradient_in_one_pass(n, m, B, T, scale):
    p = synth.gru_params(n, m, seed=21, tag="g/gru")
    x = synth.x_gaussian(B, T, m, seed=21, tag="g/x")
    y0 = synth.normal(21, "g/y0", (B, n)) * np.float32(0.5)
    gy = synth.normal(21, "g/gy", (B, T, n)) * np.float32(scale)
    y = oracle.gru_seq(p, x, y0, np.float32)
    got = bd.deer_gru_vjp(bd.GruParamsDev.from_numpy(p), dev(x), dev(y0), dev(y), dev(gy))
    want = oracle.gru_bptt(p, x, y0, y.astype(np.float64), gy.astype(np.float64), np.float64)
    for k in ("dW_i", "dW_h", "db_i", "db_h", "dx", "dy0"):
        a, b = got[k].cpu().numpy().astype(np.float64), want[k]
        # the adjoint's boundaries (4e-6 of max|lambda| each, far less in all but the last place of a few) and gates good to
        # 3e-7; the contraction adds 2^-24 per product and 64 cuts of 2^-24 between two flushes: below 4e-6 of the norm
        assert np.linalg.norm(a - b) <= 8e-6 * np.linalg.norm(b), k


def test_gradient_in_one_pass_without_dx():
    """The sums are the same bit for bit where dx is not asked for."""
    n, m, B, T = 32, 20, 3, 1001
    p = bd.GruParamsDev.from_numpy(synth.gru_params(n, m, seed=22, tag="g/gru"))
    x, y0 = dev(synth.x_gaussian(B, T, m, seed=22, tag="g/x")), torch.zeros((B, n), device="cuda")
    y = bd.deer_gru_eval(p, x, y0).y
    gy = dev(synth.normal(22, "g/gy", (B, T, n)))
    with_dx = bd.deer_gru_vjp(p, x, y0, y, gy)
    without = bd.deer_gru_vjp(p, x, y0, y, gy, want_dx=False)
    for k in ("dW_i", "dW_h", "db_i", "db_h"):
        assert torch.equal(with_dx[k], without[k]), k


@pytest.mark.parametrize("n,m", [(16, 20), (24, 33), (32, 5), (32, 32), (64, 20), (64, 63)])
def test_infinite_gradients_stay_infinite(n, m):
    """One infinite dL/dy among sequences of one step: dx is infinite there, or a NaN where infinities of both signs meet, and
    the other positions' is what it is without."""
    p = synth.gru_params(n, m, seed=23, tag="g/gru")
    x, y0 = synth.x_gaussian(70, 1, m, seed=23, tag="g/x"), synth.normal(23, "g/y0", (70, n)) * np.float32(0.5)
    gy = synth.normal(23, "g/gy", (70, 1, n))
    gy[65, 0, 2], gy[3, 0, 1] = np.inf, -np.inf
    y = oracle.gru_seq(p, x, y0, np.float32)
    got = bd.deer_gru_vjp(bd.GruParamsDev.from_numpy(p), dev(x), dev(y0), dev(y), dev(gy))["dx"].cpu().numpy()
    with np.errstate(invalid="ignore"):
        want = oracle.gru_bptt(p, x, y0, y.astype(np.float64), gy.astype(np.float64), np.float64)["dx"]
    assert np.isinf(want).any() and np.array_equal(got[~np.isfinite(want)], want[~np.isfinite(want)].astype(np.float32), equal_nan=True)
    at = np.isfinite(want)
    assert at.sum() == 68 * m and np.linalg.norm(got[at] - want[at]) <= 8e-6 * np.linalg.norm(want[at])


@pytest.mark.parametrize("n,m", [(16, 8), (24, 33), (32, 31), (32, 64), (64, 1), (64, 6), (64, 31)])
def test_dx_is_no_further_off_than_fp32_sums(n, m):
    """Sums whose terms have one sign, so that every cut of an accumulator is on the same side: dx against the error that its
    sums have in fp32 arithmetic, in order."""
    p = synth.gru_params(n, m, seed=24, tag="g/gru")
    p.W_i[:], p.W_h[:] = np.abs(p.W_i), 0.3 * np.abs(p.W_h)
    p.W_i[2 * n:] *= np.float32(0.2)
    p.b_i[2 * n:], p.b_h[2 * n:] = -3.0, 1.0                     # dG > 0: h_prev above the candidate, W_hn h + b_hn > 0
    N = 1500
    x, h = np.float32(min(0.3, 3 / m)) * np.abs(synth.x_gaussian(N, 1, m, seed=24, tag="g/x")), np.abs(synth.normal(24, "g/y0", (N, n)))
    gy = np.abs(synth.normal(24, "g/gy", (N, 1, n))) + np.float32(0.1)
    y = oracle.gru_seq(p, x, h, np.float32)
    got = bd.deer_gru_vjp(bd.GruParamsDev.from_numpy(p), dev(x), dev(h), dev(y), dev(gy))["dx"].cpu().numpy()[:, 0]
    u, q = x[:, 0].astype(np.float64) @ p.W_i.T.astype(np.float64) + p.b_i, h.astype(np.float64) @ p.W_h.T.astype(np.float64) + p.b_h
    r, z = (1 / (1 + np.exp(-u[:, g * n:g * n + n] - q[:, g * n:g * n + n])) for g in (0, 1))
    c = np.tanh(u[:, 2 * n:] + r * q[:, 2 * n:])
    dn = gy[:, 0] * (1 - z) * (1 - c * c)
    dG = np.concatenate([dn * q[:, 2 * n:] * r * (1 - r), gy[:, 0] * (h - c) * z * (1 - z), dn], axis=1)
    assert (dG > 0).all()
    want, chain = dG @ p.W_i.astype(np.float64), np.zeros((N, m), np.float32)
    for k in range(3 * n):
        chain += dG[:, k, None].astype(np.float32) * p.W_i[k].astype(np.float32)
    off = lambda a: np.linalg.norm(a - want) / np.linalg.norm(want)
    assert off(got) <= off(chain), (off(got), off(chain))


@pytest.mark.parametrize("n,m,scale", [(16, 8, 1e-34), (32, 5, 1e-36), (32, 40, 1e-35), (64, 6, 1e-36), (64, 64, 1e-35)])
def test_small_dx_keeps_its_digits(n, m, scale):
    """Gradients whose last bf16 part is below what bf16 holds: dx has fp32's accuracy there too."""
    p = synth.gru_params(n, m, seed=25, tag="g/gru")
    x, y0 = synth.x_gaussian(100, 1, m, seed=25, tag="g/x"), synth.normal(25, "g/y0", (100, n)) * np.float32(0.5)
    gy = synth.normal(25, "g/gy", (100, 1, n)) * np.float32(scale)
    y = oracle.gru_seq(p, x, y0, np.float32)
    got = bd.deer_gru_vjp(bd.GruParamsDev.from_numpy(p), dev(x), dev(y0), dev(y), dev(gy))["dx"].cpu().numpy().astype(np.float64)
    want = oracle.gru_bptt(p, x, y0, y.astype(np.float64), gy.astype(np.float64), np.float64)["dx"]
    assert np.linalg.norm((got - want) / scale) <= 2e-6 * np.linalg.norm(want / scale)     # gates and sums 1e-6 (x: rounded to fp32's 2^-24)


@pytest.mark.parametrize("n,m", [(16, 8), (24, 33), (32, 32), (64, 6), (64, 64)])
def test_inputs_masked_with_the_lowest_value(n, m):
    """Steps whose first channel holds the type's lowest or largest value: their gates are closed or open for good, their
    pre-activation gradients zero, and the sums what the other steps give."""
    p = synth.gru_params(n, m, seed=26, tag="g/gru")
    x, y0 = synth.x_gaussian(70, 5, m, seed=26, tag="g/x"), synth.normal(26, "g/y0", (70, n)) * np.float32(0.5)
    top = np.finfo(np.float32).max
    x[3, 2, 0], x[40, 0, 0], x[69, 4, 0] = -top, top, -top
    gy = synth.normal(26, "g/gy", (70, 5, n))
    with np.errstate(over="ignore"):
        y = oracle.gru_seq(p, x, y0, np.float32)
        want = oracle.gru_bptt(p, x, y0, y.astype(np.float64), gy.astype(np.float64), np.float64)
    got = bd.deer_gru_vjp(bd.GruParamsDev.from_numpy(p), dev(x), dev(y0), dev(y), dev(gy))
    for k in ("dW_i", "dW_h", "db_i", "db_h", "dx", "dy0"):
        a, b = got[k].cpu().numpy().astype(np.float64), want[k]
        assert np.isfinite(b).all() and np.linalg.norm(a - b) <= 8e-6 * np.linalg.norm(b), k


# one run per CTA (the wait behind the last run only), several
@pytest.mark.parametrize("n,m,B,T", [(16, 8, 3, 64), (32, 33, 2, 97), (60, 7, 1, 65), (32, 32, 8, 5001), (24, 40, 10, 4001), (48, 20, 2, 15001)])
def test_expired_wait_is_reported(n, m, B, T):
    """The waits for a run's products run out and the adjoint's do not: the call says so, and the next one on the same workspace
    gives what one on another does."""
    p = bd.GruParamsDev.from_numpy(synth.gru_params(n, m, seed=27, tag="g/gru"))
    x, y0 = dev(synth.x_gaussian(B, T, m, seed=27, tag="g/x")), torch.zeros((B, n), device="cuda")
    y, gy = bd.deer_gru_eval(p, x, y0).y, dev(synth.normal(27, "g/gy", (B, T, n)))
    want, ws = bd.deer_gru_vjp(p, x, y0, y, gy), bd.alloc_workspace(bd.DEER_OP_VJP, B, T, n, m)
    for flags in (bd.DEER_FLAG_EXPIRE_PRODUCT_WAITS, 0):
        got = bd.deer_gru_vjp(p, x, y0, y, gy, ws=ws, flags=flags)
        assert bd.deer_workspace_status(ws) == (bd.DEER_ERR_DEVICE_TIMEOUT if flags else bd.DEER_OK)
    for k, v in want.items():
        assert torch.equal(got[k], v), k
