"""Chains with a verified burn-in (bodies, adjoints and stand-alone scans as one launch each) at the sizes where they can go
wrong: remainders of chains, tiles and CTAs, the ends of a dispatch range, inputs and cells for which a burn-in is raised or
the launch gives up.  Every case states the kernel it is meant for, and that kernel has to have run."""
import numpy as np
import pytest
import torch

import oracle
from paper_2309_12252_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bd():
    from paper_2309_12252_b200 import binding
    binding.lib()
    return binding


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def launched(bd, call):
    """The call's result and the names of the kernels that it launched."""
    from bench import read_profile
    bd.lib().deer_profile_enable(1)
    try:
        r = call()
        torch.cuda.synchronize()
    finally:
        bd.lib().deer_profile_enable(0)
    return r, set(read_profile(bd))


def walk(x):
    x = np.cumsum(x.astype(np.float64), axis=1)
    return ((x - x.mean(1, keepdims=True)) / x.std(1, keepdims=True)).astype(np.float32)


def behind(names):
    """Did the kernels that multiply the Jacobians out do a body?"""
    return any(k.startswith("cell_") for k in names)


def projected(names):
    return bool(names & {"proj_tiled_kernel", "affine_mma_kernel"})


SEG, ONE, TILE, LANE = "newton_segment_kernel", "newton_body_kernel", "newton_tile_kernel", "newton_lane_kernel"


@pytest.mark.parametrize("n,m,B,T,x_kind,kernel", [
    (1, 1, 1, 3, "noise", SEG), (3, 70, 2, 129, "noise", SEG), (12, 5, 3, 401, "walk", SEG), (31, 3, 1, 80, "noise", SEG),
    (32, 64, 2, 97, "walk", SEG), (40, 7, 2, 51, "noise", SEG),
    (16, 3, 16, 5001, "noise", SEG), (24, 10, 16, 6001, "noise", SEG),                       # a launch per body
    (16, 5, 16, 15001, "noise", ONE), (50, 1, 4, 663, "noise", ONE), (43, 64, 5, 2003, "walk", ONE),
    (32, 33, 16, 6001, "noise", TILE), (32, 3, 3, 40001, "walk", TILE), (32, 64, 17, 16001, "noise", TILE),
    (64, 1, 1, 16001, "noise", TILE), (64, 64, 7, 2801, "walk", TILE),
    (1, 1, 16, 300001, "noise", LANE), (3, 2, 5, 50001, "noise", LANE), (4, 3, 16, 50003, "noise", LANE), (5, 9, 16, 20001, "walk", LANE),
    (8, 8, 16, 30001, "noise", LANE), (2, 2, 16, 100001, "walk", None)])
def test_bodies(bd, n, m, B, T, x_kind, kernel):
    p = synth.gru_params(n, m, seed=3, tag="c/gru")
    x = synth.x_gaussian(B, T, m, seed=3, tag="c/x")
    if x_kind == "walk":
        x = walk(x)
    y0 = synth.normal(3, "c/y0", (B, n)) * 0.5
    pd, xd, yd = bd.GruParamsDev.from_numpy(p), dev(x), dev(y0)
    r, names = launched(bd, lambda: bd.deer_gru_eval(pd, xd, yd))
    assert kernel is None or kernel in names, names
    assert r.status == 0 and r.err <= 1e-4
    assert np.max(np.abs(r.y.cpu().numpy() - oracle.gru_seq(p, x, y0, np.float32))) <= 1e-4


@pytest.mark.parametrize("n,m,B,T,bias,warm,kernel", [
    (8, 4, 16, 9001, 0.0, False, SEG), (8, 4, 16, 9001, 1.0, False, SEG), (24, 5, 2, 3001, 1.0, False, SEG), (24, 5, 2, 3001, 0.0, True, SEG),
    (16, 5, 16, 15001, 1.0, False, ONE), (32, 33, 16, 6001, 1.0, False, TILE), (64, 3, 3, 12001, 0.0, False, TILE),
    (64, 3, 3, 12001, 1.0, False, TILE), (64, 3, 3, 12001, 0.0, True, TILE)])
def test_burn_in_of_each_body_follows_the_cell(bd, n, m, B, T, bias, warm, kernel):
    """Short chains take the burn-in that their last body's mismatch calls for: cells that forget fast and slowly (update gates
    biased to keep), and a guess that is near the solution, whose first update asks for more than a twentieth.  Every boundary of
    the last body is good to 2.4e-7 or a thousandth of the tolerance, the gates to 2e-7, and a cell that forgets a tenth a step
    carries ten times that."""
    p = synth.gru_params(n, m, seed=6, tag="c/gru")
    p.b_i[n:2 * n] += bias
    x = synth.x_gaussian(B, T, m, seed=6, tag="c/x")
    y0 = synth.normal(6, "c/y0", (B, n)) * 0.5
    want = oracle.gru_seq(p, x, y0, np.float32)
    args = bd.GruParamsDev.from_numpy(p), dev(x), dev(y0)
    y = dev(want + 1e-2 * synth.normal(6, "c/guess", want.shape)) if warm else None
    r, names = launched(bd, lambda: bd.deer_gru_eval(*args, y=y, flags=bd.DEER_FLAG_WARM_START if warm else 0))
    # (of the cells that keep more, those of n = 16 and 32 ask for more than is worth trying beside the kernels behind)
    assert kernel in names and behind(names) == (bias > 0 and n in (16, 32)), names
    assert r.status == 0 and r.err <= 1e-4
    assert np.max(np.abs(r.y.cpu().numpy() - want)) <= 1e-5
    if not warm:
        exact = bd.deer_gru_eval(*args, flags=bd.DEER_FLAG_MATERIALIZE)
        assert abs(r.iters - exact.iters) <= 1, (r.iters, exact.iters)


@pytest.mark.parametrize("n,m,B,T,bias", [(8, 4, 16, 9001, 2.5), (8, 4, 16, 9001, 2.2), (5, 3, 4, 4001, 2.6), (24, 5, 2, 3001, 2.4), (40, 7, 2, 1501, 2.2)])
@pytest.mark.parametrize("off", [1e-2, 5e-2])
def test_warm_start_of_a_cell_that_forgets_a_tenth_a_step(bd, n, m, B, T, bias, off):
    """The first update is small and calls for some hundred steps of burn-in, as many as the two-phase form's shared memory holds
    or a few more.  (Gates good to 2e-7 and boundaries to a thousandth of the tolerance, carried over some twenty steps.)"""
    p = synth.gru_params(n, m, seed=6, tag="c/gru")
    p.b_i[n:2 * n] += np.float32(bias)
    x = synth.x_gaussian(B, T, m, seed=6, tag="c/x")
    y0 = synth.normal(6, "c/y0", (B, n)) * 0.5
    want = oracle.gru_seq(p, x, y0, np.float32)
    y = dev(want + off * synth.normal(6, "c/guess", want.shape))
    r, names = launched(bd, lambda: bd.deer_gru_eval(bd.GruParamsDev.from_numpy(p), dev(x), dev(y0), y=y, flags=bd.DEER_FLAG_WARM_START))
    assert SEG in names, names
    assert r.status == 0 and r.err <= 1e-4
    assert np.max(np.abs(r.y.cpu().numpy() - want)) <= 2e-5


@pytest.mark.parametrize("n,m,B,T", [(1, 1, 16, 300001), (8, 4, 4, 1000), (16, 8, 8, 20000), (24, 3, 2, 700), (32, 8, 16, 8000), (64, 6, 2, 9000)])
def test_cell_that_remembers_for_long(bd, n, m, B, T):
    """The update gate's bias alone keeps the state: no burn-in is tried, the Jacobians are multiplied out."""
    p = synth.gru_params(n, m, seed=4, tag="c/gru")
    p.b_i[n:2 * n] += 6.0
    x = synth.x_gaussian(B, T, m, seed=4, tag="c/x")
    y0 = synth.normal(4, "c/y0", (B, n)) * 0.5
    r = bd.deer_gru_eval(bd.GruParamsDev.from_numpy(p), dev(x), dev(y0))
    assert r.status == 0
    assert np.max(np.abs(r.y.cpu().numpy() - oracle.gru_seq(p, x, y0, np.float32))) <= 1e-3


WARP, MMA_TILE, ROWS = "newton_adjoint_kernel", "adjoint_tile_kernel", "rows_adjoint_kernel"


@pytest.mark.parametrize("n,m,B,T,dense,x_kind,kernel", [
    (3, 7, 2, 5001, True, "noise", WARP), (12, 5, 8, 3001, True, "walk", WARP), (9, 60, 4, 15001, True, "noise", WARP),
    (16, 8, 16, 20001, True, "noise", WARP), (24, 3, 1, 6001, False, "noise", WARP), (32, 32, 16, 10001, True, "walk", WARP),
    (40, 7, 2, 4001, False, "noise", WARP), (56, 1, 3, 3001, True, "noise", WARP),
    (64, 6, 3, 20001, True, "walk", MMA_TILE), (64, 64, 16, 4003, False, "noise", MMA_TILE),
    (1, 8, 5, 20003, True, "noise", ROWS), (8, 1, 1, 45, False, "walk", ROWS), (2, 4, 64, 67, True, "noise", ROWS)])
def test_adjoints(bd, n, m, B, T, dense, x_kind, kernel):
    p = synth.gru_params(n, m, 5, tag="c/gru")
    x = synth.x_gaussian(B, T, m, 5, tag="c/x")
    if x_kind == "walk":
        x = walk(x)
    y0 = synth.normal(5, "c/y0", (B, n)) * 0.3
    y = oracle.gru_seq(p, x, y0, np.float32)
    gy = synth.normal(5, "c/gy", (B, T, n))
    if not dense:                      # a loss on the last step: dy0 is far below max|lambda|
        gy[:, :-1] = 0.0
    want = oracle.gru_bptt(p, x, y0, y.astype(np.float64), gy, np.float64)
    args = bd.GruParamsDev.from_numpy(p), dev(x), dev(y0), dev(y), dev(gy)
    got, names = launched(bd, lambda: bd.deer_gru_vjp(*args, want_dx=True))
    assert kernel in names, names
    for k in ("dW_i", "dW_h", "db_i", "db_h", "dx", "dy0"):
        a, b = got[k].cpu().numpy().astype(np.float64), want[k]
        assert np.max(np.abs(a - b)) <= 1e-3 * max(np.max(np.abs(b)), 1e-30), k


@pytest.mark.parametrize("n,B,T", [(4, 2, 65537), (8, 3, 60001), (16, 1, 9001), (32, 2, 1111), (32, 16, 1300), (64, 1, 515), (64, 5, 193)])
@pytest.mark.parametrize("reverse", [False, True])
@pytest.mark.parametrize("decays", [True, False])
def test_scans(bd, n, B, T, reverse, decays):
    """Matrices whose products hardly decay make the boundaries differ: the chunked scan behind does the work."""
    J = synth.contractive_J(B, T, n, seed=n + T, tag="c/J", scale=1.0)
    if not decays:
        J = 0.05 * J + 0.95 * np.eye(n, dtype=np.float32) * np.float32(1.04)
    b = synth.normal(n + T, "c/b", (B, T, n))
    y0 = synth.normal(n + T, "c/y0", (B, n))
    want = oracle.linrec(J, b, y0, reverse=reverse, dtype=np.float64)
    args = dev(J), dev(b), dev(y0)
    got, names = launched(bd, lambda: bd.deer_linrec_scan(*args, reverse=reverse))
    assert "scan_verified_kernel" in names, names
    tol = 1e-5 if decays else 1e-4     # (sums over some eighty positions instead of two)
    assert np.max(np.abs(got.cpu().numpy() - want)) <= tol * max(1.0, float(np.max(np.abs(want))))


@pytest.mark.parametrize("n,B,T", [(4, 2, 65537), (8, 3, 60001), (16, 1, 9001), (32, 16, 1300), (64, 1, 515)])
@pytest.mark.parametrize("reverse", [False, True])
def test_scan_components_of_unequal_size(bd, n, B, T, reverse):
    """Every other component is large and forgets at once, the ones between are 1e9 times smaller and remember: each is good to
    fp32 in its own size (sums over some hundred positions: a hundred roundings of 6e-8, six of them allowed for each)."""
    J = np.zeros((B, T, n, n), np.float32)
    i = np.arange(n)
    J[:, :, i, i] = np.where(i % 2 == 0, 0.5, 0.99)
    b = synth.normal(n + T, "c/b", (B, T, n)) * np.where(i % 2 == 0, 1e6, 1e-3).astype(np.float32)
    want = oracle.linrec(J, b, None, reverse=reverse, dtype=np.float64)
    args = dev(J), dev(b)
    got, names = launched(bd, lambda: bd.deer_linrec_scan(*args, reverse=reverse))
    assert "scan_verified_kernel" in names, names
    off = np.max(np.abs(got.cpu().numpy() - want), axis=(0, 1)) / np.max(np.abs(want), axis=(0, 1))
    assert np.max(off) <= 4e-5, off


def accepted(ws):
    """StatusBlock::done of the call that last used the workspace: set where a launch with verified boundaries did the work."""
    return int(ws[:16].view(torch.int32)[3].item())


@pytest.mark.parametrize("n,m,B,T", [(50, 70, 4, 5000), (56, 100, 6, 4003), (64, 65, 8, 30001)])
def test_adjoint_of_wide_states_with_projected_inputs(bd, n, m, B, T):
    """Chains of four positions: the start states of all of them have room beside the projected inputs that the launch and the
    kernels behind it read."""
    p = synth.gru_params(n, m, 6, tag="c/gru")
    x = synth.x_gaussian(B, T, m, 6, tag="c/x")
    y0 = synth.normal(6, "c/y0", (B, n)) * 0.3
    y = oracle.gru_seq(p, x, y0, np.float32)
    gy = synth.normal(6, "c/gy", (B, T, n))
    want = oracle.gru_bptt(p, x, y0, y.astype(np.float64), gy, np.float64)
    args = bd.GruParamsDev.from_numpy(p), dev(x), dev(y0), dev(y), dev(gy)
    ws = bd.alloc_workspace(bd.DEER_OP_VJP, B, T, n, m)
    got, names = launched(bd, lambda: bd.deer_gru_vjp(*args, want_dx=True, ws=ws))
    assert WARP in names and accepted(ws) == 1, names
    for k in ("dW_i", "dW_h", "db_i", "db_h", "dx", "dy0"):
        a, b = got[k].cpu().numpy().astype(np.float64), want[k]
        assert np.max(np.abs(a - b)) <= 1e-3 * np.max(np.abs(b)), k


@pytest.mark.parametrize("n,m,B,T", [(8, 8, 64, 1000), (8, 1, 3, 4001), (8, 4, 16, 2300), (4, 2, 33, 701), (2, 1, 9, 500), (1, 4, 40, 777)])
def test_adjoint_of_small_cells_in_short_chains(bd, n, m, B, T):
    """Chains of four or eight positions, a boundary per four to thirty-two of them: all are told apart, and the launch's result
    is taken."""
    p = synth.gru_params(n, m, 7, tag="c/gru")
    x = synth.x_gaussian(B, T, m, 7, tag="c/x")
    y0 = synth.normal(7, "c/y0", (B, n)) * 0.3
    y = oracle.gru_seq(p, x, y0, np.float32)
    gy = synth.normal(7, "c/gy", (B, T, n))
    want = oracle.gru_bptt(p, x, y0, y.astype(np.float64), gy, np.float64)
    args = bd.GruParamsDev.from_numpy(p), dev(x), dev(y0), dev(y), dev(gy)
    ws = bd.alloc_workspace(bd.DEER_OP_VJP, B, T, n, m)
    got, names = launched(bd, lambda: bd.deer_gru_vjp(*args, want_dx=True, ws=ws))
    assert ROWS in names and accepted(ws) == 1, names
    for k in ("dW_i", "dW_h", "db_i", "db_h", "dx", "dy0"):
        a, b = got[k].cpu().numpy().astype(np.float64), want[k]
        assert np.max(np.abs(a - b)) <= 1e-4 * np.max(np.abs(b)), k


def gradient(bd, p, x, y0, gy, **kw):
    """deer_gru_vjp at the sequential trajectory, the fp64 gradients, the kernels launched, whether their result was taken."""
    y = oracle.gru_seq(p, x, y0, np.float32)
    want = oracle.gru_bptt(p, x, y0, y.astype(np.float64), gy, np.float64)
    args = bd.GruParamsDev.from_numpy(p), dev(x), dev(y0), dev(y), dev(gy)
    B, T, m = x.shape
    ws = bd.alloc_workspace(bd.DEER_OP_VJP, B, T, p.b_i.size // 3, m)
    got, names = launched(bd, lambda: bd.deer_gru_vjp(*args, want_dx=True, ws=ws, **kw))
    got = {k: v.cpu().numpy().astype(np.float64) for k, v in got.items() if v is not None}
    return got, want, names, accepted(ws)


SCALES = [(8, 4, 16, 10001, ROWS), (2, 1, 16, 40001, ROWS), (24, 3, 2, 6001, WARP), (32, 8, 16, 9001, WARP), (64, 6, 4, 20001, MMA_TILE)]


@pytest.mark.parametrize("n,m,B,T,kernel", SCALES)
def test_adjoint_of_sequences_of_unequal_weight(bd, n, m, B, T, kernel):
    """The first sequence's loss weighs most and its inputs make the cell forget; the others weigh a millionth or less and
    remember.  Each has its own dx and dy0 to a thousandth, the tolerance that gradients have everywhere."""
    p = synth.gru_params(n, m, 8, tag="c/gru")
    p.W_i[n:2 * n, 0] = 1.0
    x = synth.x_gaussian(B, T, m, 8, tag="c/x")
    x[:, :, 0] = 2.0 + 0.25 * x[:, :, 0]
    x[0, :, 0] -= 6.0
    y0 = synth.normal(8, "c/y0", (B, n)) * 0.3
    gy = synth.normal(8, "c/gy", (B, T, n))
    gy[1::2] *= np.float32(1e-6)
    gy[2::2] *= np.float32(1e-12)
    got, want, names, _ = gradient(bd, p, x, y0, gy)
    assert kernel in names, names
    for k in ("dx", "dy0"):
        for b in range(B):
            assert np.max(np.abs(got[k][b] - want[k][b])) <= 1e-3 * np.max(np.abs(want[k][b])), (k, b)


@pytest.mark.parametrize("n,m,B,T,kernel", SCALES)
def test_adjoint_behind_a_loss_on_the_last_step(bd, n, m, B, T, kernel):
    """lambda decays through every magnitude towards the first step: dx is right at each, compared in blocks of eight steps as
    long as it is an ordinary fp32 number (products of up to some hundred Jacobians, each good to about 1e-5)."""
    p = synth.gru_params(n, m, 9, tag="c/gru")
    x = synth.x_gaussian(B, T, m, 9, tag="c/x")
    y0 = synth.normal(9, "c/y0", (B, n)) * 0.3
    gy = np.zeros((B, T, n), np.float32)
    gy[:, -1] = synth.normal(9, "c/gy", (B, n))
    got, want, names, _ = gradient(bd, p, x, y0, gy)
    assert kernel in names, names
    blocks = 0
    for b in range(B):
        for t in range(T - 8, T - 400, -8):
            top = np.max(np.abs(want["dx"][b, t:t + 8]))
            if top < 1e-25:
                break
            assert np.max(np.abs(got["dx"][b, t:t + 8] - want["dx"][b, t:t + 8])) <= 1e-2 * top, (b, T - t)
            blocks += 1
    assert blocks > 6 * B              # (n = 2 decays by 1e-25 within some sixty steps)


@pytest.mark.parametrize("t", [0, 1, 1000, 12000])
def test_adjoint_tile_beyond_the_range_of_its_operands(bd, t):
    """Inputs that f16 halves cannot hold make the tile's result a NaN, at the first time step only in the gradients there: the
    launch has to see it whether dy0 is wanted or not, and the kernels behind do the work."""
    n, m, B, T = 64, 6, 5, 12001
    p = synth.gru_params(n, m, 10, tag="c/gru")
    x = synth.x_gaussian(B, T, m, 10, tag="c/x")
    x[1, t] *= np.float32(2e4)
    gy = synth.normal(10, "c/gy", (B, T, n))
    for want_dy0 in (False, True):
        got, want, names, done = gradient(bd, p, x, np.zeros((B, n), np.float32), gy, want_dy0=want_dy0)
        assert MMA_TILE in names and done == 0, names
        for k in got:
            assert np.max(np.abs(got[k] - want[k])) <= 1e-3 * np.max(np.abs(want[k])), k


@pytest.mark.parametrize("n,m,B,T,kernel", [(4, 2, 1, 1000, SEG), (24, 10, 5, 1001, SEG), (32, 33, 16, 6001, TILE), (64, 6, 3, 9001, TILE)])
def test_expired_wait_in_a_body_is_reported(bd, n, m, B, T, kernel):
    """The whole-loop kernel's wait for the other CTAs and the tile's for its products are bounded: where one runs out the
    evaluation says so, and the next call on the same workspace is right."""
    p = synth.gru_params(n, m, seed=11, tag="c/gru")
    x = synth.x_gaussian(B, T, m, seed=11, tag="c/x")
    y0 = synth.normal(11, "c/y0", (B, n)) * 0.5
    pd, xd, yd = bd.GruParamsDev.from_numpy(p), dev(x), dev(y0)
    ws = bd.alloc_workspace(bd.DEER_OP_EVAL, B, T, n, m)
    r, names = launched(bd, lambda: bd.deer_gru_eval(pd, xd, yd, ws=ws, flags=bd.DEER_FLAG_EXPIRE_BODY_WAITS, check=False))
    assert kernel in names and r.status == bd.DEER_ERR_DEVICE_TIMEOUT, (names, r.status)
    r = bd.deer_gru_eval(pd, xd, yd, ws=ws)
    assert r.status == 0
    assert np.max(np.abs(r.y.cpu().numpy() - oracle.gru_seq(p, x, y0, np.float32))) <= 1e-4


def test_expired_wait_in_the_adjoint_tile_is_reported(bd):
    n, m, B, T = 64, 6, 5, 12001
    p = synth.gru_params(n, m, seed=12, tag="c/gru")
    x = synth.x_gaussian(B, T, m, seed=12, tag="c/x")
    y0 = np.zeros((B, n), np.float32)
    gy = synth.normal(12, "c/gy", (B, T, n))
    y = oracle.gru_seq(p, x, y0, np.float32)
    args = bd.GruParamsDev.from_numpy(p), dev(x), dev(y0), dev(y), dev(gy)
    ws = bd.alloc_workspace(bd.DEER_OP_VJP, B, T, n, m)
    _, names = launched(bd, lambda: bd.deer_gru_vjp(*args, ws=ws, flags=bd.DEER_FLAG_EXPIRE_BODY_WAITS))
    assert MMA_TILE in names and accepted(ws) == 0
    assert bd.deer_workspace_status(ws) == bd.DEER_ERR_DEVICE_TIMEOUT
    got = bd.deer_gru_vjp(*args, ws=ws)
    assert accepted(ws) == 1 and bd.deer_workspace_status(ws) == bd.DEER_OK
    want = oracle.gru_bptt(p, x, y0, y.astype(np.float64), gy, np.float64)
    assert np.max(np.abs(got["dW_h"].cpu().numpy() - want["dW_h"])) <= 1e-3 * np.max(np.abs(want["dW_h"]))


def test_expired_wait_in_the_multihead_loop_is_reported(bd):
    H, n, m, B, T = 3, 8, 5, 2, 300
    heads = [bd.GruParamsDev.from_numpy(synth.gru_params(n, m, seed=h, tag="c/gru")) for h in range(H)]
    x, y0 = dev(synth.x_gaussian(B, T, m, seed=13, tag="c/x")), torch.zeros((B, H, n), device="cuda")
    with pytest.raises(bd.DeerError):
        bd.deer_gru_multihead_eval(heads, [1, 2, 4], x, y0, flags=bd.DEER_FLAG_EXPIRE_BODY_WAITS)
    assert bd.deer_gru_multihead_eval(heads, [1, 2, 4], x, y0)[2] == 0


@pytest.mark.parametrize("n,m,B,T,bias", [(16, 8, 4, 30000, 6.0), (8, 4, 16, 60000, 6.0), (8, 4, 16, 60000, 0.0), (32, 8, 16, 40000, 0.0)])
def test_host_call_copies_finished_results_only(bd, n, m, B, T, bias):
    """The selection of the current iterate goes before a copy of a result to host memory: one per chunk of the call at most,
    whatever forms give up and however many groups of bodies the loop takes."""
    p = synth.gru_params(n, m, seed=14, tag="c/gru")
    p.b_i[n:2 * n] += np.float32(bias)
    x = walk(synth.x_gaussian(B, T, m, seed=14, tag="c/x"))
    pd, y0, xd, yd = bd.GruParamsDev.from_numpy(p), torch.zeros((B, n), device="cuda"), torch.empty((B, T, m), device="cuda"), torch.empty((B, T, n), device="cuda")
    xh, yh = torch.from_numpy(x).pin_memory(), torch.empty((B, T, n), pin_memory=True)
    ws = bd.alloc_workspace(bd.DEER_OP_EVAL, B, T, n, m)
    from bench import read_profile
    bd.lib().deer_profile_enable(1)
    try:
        bd.deer_gru_eval_host(pd, xh, y0, yh, xd, yd, ws)
    finally:
        bd.lib().deer_profile_enable(0)
    first = bd.deer_gru_eval_host_chunks(B, T)
    assert read_profile(bd).get("result_select_kernel", {"launches": 0})["launches"] <= len(first) - 1
    for lo, hi in zip(first[:-1], first[1:]):          # (bit for bit, also where the iteration of a cell that remembers diverges)
        alone = bd.deer_gru_eval(pd, dev(x[lo:hi]), y0[lo:hi].contiguous())
        assert np.array_equal(yh.numpy()[lo:hi], alone.y.cpu().numpy(), equal_nan=True)


# ---- the launches are not only made but taken: the kernels behind them do nothing, and the accuracy is the launches' own
@pytest.mark.parametrize("n,m,B,T,kernel", [
    (1, 1, 1, 400, SEG), (3, 70, 2, 129, SEG), (12, 5, 3, 401, SEG), (32, 64, 2, 97, SEG), (40, 7, 2, 51, SEG), (24, 10, 16, 6001, SEG),
    (16, 5, 16, 15001, ONE), (50, 1, 4, 663, ONE), (43, 64, 5, 2003, ONE),
    (32, 33, 16, 6001, TILE), (32, 3, 3, 40001, TILE), (32, 64, 17, 16001, TILE), (64, 1, 1, 16001, TILE), (64, 64, 7, 2801, TILE),
    (1, 1, 16, 300001, LANE), (3, 2, 5, 50001, LANE), (4, 3, 16, 50003, LANE), (5, 9, 16, 20001, LANE), (8, 8, 16, 30001, LANE)])
def test_bodies_are_taken(bd, n, m, B, T, kernel):
    p = synth.gru_params(n, m, seed=15, tag="c/gru")
    x = synth.x_gaussian(B, T, m, seed=15, tag="c/x")
    y0 = synth.normal(15, "c/y0", (B, n)) * 0.5
    pd, xd, yd = bd.GruParamsDev.from_numpy(p), dev(x), dev(y0)
    r, names = launched(bd, lambda: bd.deer_gru_eval(pd, xd, yd))
    assert {k for k in names if k.startswith("newton_")} == {kernel}, names
    assert not any(k.startswith(("cell_", "scan_", "gen_")) for k in names), names
    assert r.status == 0 and r.err <= 1e-4
    assert np.max(np.abs(r.y.cpu().numpy() - oracle.gru_seq(p, x, y0, np.float32))) <= 1e-5     # (quadratic: far below the last update)


@pytest.mark.parametrize("n,m,B,T,x_kind,kernel", [
    (3, 7, 2, 5001, "noise", WARP), (12, 5, 8, 3001, "noise", WARP), (9, 60, 4, 15001, "noise", WARP), (16, 8, 16, 20001, "noise", WARP),
    (32, 32, 16, 10001, "noise", WARP), (40, 7, 2, 9001, "noise", WARP), (56, 1, 3, 9001, "noise", WARP),
    (64, 6, 3, 20001, "noise", MMA_TILE), (64, 64, 16, 4003, "noise", MMA_TILE),
    (1, 8, 5, 20003, "noise", ROWS), (8, 1, 1, 45, "noise", ROWS), (2, 4, 64, 67, "noise", ROWS), (8, 8, 16, 30001, "noise", ROWS)])
def test_adjoints_are_taken(bd, n, m, B, T, x_kind, kernel):
    """Boundaries within 4e-6 of max|lambda| and products of fp32 level: 2e-5 of the largest entry of dx and dy0, and of sums over
    all positions."""
    p = synth.gru_params(n, m, 16, tag="c/gru")
    x = synth.x_gaussian(B, T, m, 16, tag="c/x")
    y0 = synth.normal(16, "c/y0", (B, n)) * 0.3
    gy = synth.normal(16, "c/gy", (B, T, n))
    got, want, names, done = gradient(bd, p, x, y0, gy)
    assert kernel in names and done == 1, names
    for k in ("dW_i", "dW_h", "db_i", "db_h", "dx", "dy0"):
        assert np.max(np.abs(got[k] - want[k])) <= 2e-5 * np.max(np.abs(want[k])), k


@pytest.mark.parametrize("n,B,T", [(4, 2, 65537), (8, 3, 60001), (16, 1, 9001), (32, 2, 1111), (32, 16, 1300), (64, 1, 515), (64, 5, 193)])
@pytest.mark.parametrize("reverse", [False, True])
@pytest.mark.parametrize("decays", [True, False])
def test_scans_are_taken_where_products_decay(bd, n, B, T, reverse, decays):
    J = synth.contractive_J(B, T, n, seed=n + T, tag="c/J", scale=1.0)
    if not decays:
        J = 0.05 * J + 0.95 * np.eye(n, dtype=np.float32) * np.float32(1.04)
    ws = bd.alloc_workspace(bd.DEER_OP_SCAN, B, T, n)
    bd.deer_linrec_scan(dev(J), dev(synth.normal(n + T, "c/b", (B, T, n))), dev(synth.normal(n + T, "c/y0", (B, n))), reverse=reverse, ws=ws)
    assert accepted(ws) == int(decays)


@pytest.mark.parametrize("n,m,B,T", [(32, 32, 16, 6001), (64, 6, 3, 9001)])
@pytest.mark.parametrize("t", [0, 3000, 5999])
def test_evaluation_tile_beyond_the_range_of_its_operands(bd, n, m, B, T, t):
    """An input that f16 halves cannot hold: the tiles give up and the kernels behind do the work."""
    p = synth.gru_params(n, m, 17, tag="c/gru")
    x = synth.x_gaussian(B, T, m, 17, tag="c/x")
    x[1, t] *= np.float32(2e4)
    y0 = synth.normal(17, "c/y0", (B, n)) * 0.5
    r, names = launched(bd, lambda: bd.deer_gru_eval(bd.GruParamsDev.from_numpy(p), dev(x), dev(y0)))
    assert TILE in names and behind(names), names
    assert r.status == 0
    assert np.max(np.abs(r.y.cpu().numpy() - oracle.gru_seq(p, x, y0, np.float32))) <= 1e-4


@pytest.mark.parametrize("n,m,B,T", [(32, 32, 16, 6001), (64, 6, 3, 9001)])
@pytest.mark.parametrize("scale", [1.0, 1e-2, 1e-4])
def test_evaluation_tile_on_small_inputs(bd, n, m, B, T, scale):
    """Operands are good to 2^-23 of themselves and, below 2^-6, to 2^-29 absolute.  Without biases the states are as small as the
    inputs: m + n such errors, weighted by up to 1 / sqrt(n), the 2e-7 absolute of the gates' tanh (half of it with z about 1/2),
    both summed over some four steps of memory, beside fp32 rounding.  The tanh leads, as it does in the kernels that multiply
    the Jacobians out: the tile is no further off than they are, but for its operands."""
    p = synth.gru_params(n, m, 18, tag="c/gru")
    p.b_i[:] = 0.0
    p.b_h[:] = 0.0
    x = synth.x_gaussian(B, T, m, 18, tag="c/x") * np.float32(scale)
    y0 = np.zeros((B, n), np.float32)
    args = bd.GruParamsDev.from_numpy(p), dev(x), dev(y0)
    r, names = launched(bd, lambda: bd.deer_gru_eval(*args, tol=-1.0, max_iter=6))
    assert TILE in names, names
    want = oracle.gru_seq(p, x, y0, np.float64)
    operands, rounding = 4.0 * (m + n) * 2.0 ** -29 / np.sqrt(n), 4e-6 * np.max(np.abs(want))
    off = np.max(np.abs(r.y.cpu().numpy() - want))
    assert off <= operands + 4.0 * 1e-7 + rounding
    other, names = launched(bd, lambda: bd.deer_gru_eval(*args, tol=-1.0, max_iter=6, flags=bd.DEER_FLAG_MATERIALIZE))
    assert TILE not in names, names
    assert off <= operands + 1.5 * np.max(np.abs(other.y.cpu().numpy() - want)) + rounding / 4.0


def test_scan_of_unequal_but_coupled_components_is_taken(bd):
    """The gradient of a mean over slowly varying sequences: lambda's components differ by orders of magnitude but feed each other,
    and no fp32 sum has the small ones to more than the large ones' rounding."""
    n, m, B, T = 64, 4, 8, 2179
    p = synth.gru_params(n, m, 19, tag="c/gru")
    x = walk(synth.x_gaussian(B, T, m, 19, tag="c/x"))
    gy = np.repeat(synth.normal(19, "c/gy", (B, 1, n)) * np.float32(1.0 / T), T, axis=1)
    gy[:, :, ::2] *= np.float32(1e-4)
    got, want, names, done = gradient(bd, p, x, np.zeros((B, n), np.float32), gy)
    assert "scan_verified_kernel" in names and not names & {WARP, MMA_TILE} and done == 1, names
    for k in ("dW_i", "dW_h", "db_i", "db_h", "dx", "dy0"):
        assert np.max(np.abs(got[k] - want[k])) <= 2e-5 * np.max(np.abs(want[k])), k


@pytest.mark.parametrize("n,m,B,T,gy_scale,x_scale,kernel", [
    (9, 3, 40, 700, 1.0, 1.0, WARP), (16, 3, 16, 10001, 1.0, 1.0, WARP), (17, 16, 16, 700, 1.0, 1.0, WARP), (24, 33, 16, 700, 1e-25, 1.0, WARP),
    (32, 1, 16, 8001, 1e25, 1.0, WARP), (33, 64, 16, 1000, 1.0, 1.0, WARP), (48, 2, 16, 500, 1.0, 1.0, WARP), (57, 15, 16, 300, 1.0, 1.0, WARP),
    (63, 8, 16, 300, 1.0, 1.0, WARP), (24, 4, 16, 700, 1.0, 3000.0, WARP), (24, 4, 16, 700, 1.0, 2e4, WARP), (24, 4, 16, 700, 1.0, 4e4, None),
    (8, 16, 16, 30001, 1.0, 1.0, WARP)])
def test_adjoint_products_are_at_fp32_level(bd, n, m, B, T, gy_scale, x_scale, kernel):
    """K steps of 16 with and without their second half, gradients of any magnitude, inputs up to and beyond what the products'
    halves hold.  A product is good to 2^-22 of its operands and a lambda carries the errors of some ten steps: 2-norms agree to
    1e-6.  (An input beyond the halves' range is for the kernels behind, and saturates the gates: their 1e-3.)"""
    p = synth.gru_params(n, m, 8, tag="c/gru")
    x = synth.x_gaussian(B, T, m, 8, tag="c/x")
    x[:, :, 0] = np.clip(x[:, :, 0], -4, 4) * np.float32(x_scale)
    y0 = synth.normal(8, "c/y0", (B, n)) * 0.3
    gy = (synth.normal(8, "c/gy", (B, T, n)).astype(np.float64) * gy_scale).astype(np.float32)
    got, want, names, done = gradient(bd, p, x, y0, gy)
    assert WARP in names and done == (0 if kernel is None else 1), names
    for k in ("db_i", "db_h", "dx", "dy0"):
        a, b = got[k], want[k].astype(np.float64)
        assert np.linalg.norm(a - b) <= (1e-6 if x_scale == 1.0 else 1e-3) * np.linalg.norm(b), k


@pytest.mark.parametrize("n,m,B,T,x_scale,y0_scale,kernel", [
    (16, 5, 16, 15001, 1.0, 0.5, ONE), (12, 16, 16, 40001, 1.0, 0.5, ONE), (49, 17, 4, 663, 1.0, 0.5, ONE), (50, 33, 4, 663, 1.0, 0.5, ONE),
    (57, 15, 3, 401, 1.0, 0.5, ONE), (62, 70, 4, 300, 1.0, 0.5, ONE), (50, 3, 4, 663, 3000.0, 0.5, ONE), (50, 3, 4, 663, 2e4, 0.5, None),
    (50, 3, 4, 663, 1.0, 3.0, ONE)])
def test_one_phase_products_are_at_fp32_level(bd, n, m, B, T, x_scale, y0_scale, kernel):
    """K steps of 16 with and without their second half, and inputs and states up to and beyond what the products' halves hold.  The
    gates are good to 2e-7 and a cell as initialised carries less than ten times that."""
    p = synth.gru_params(n, m, seed=9, tag="c/gru")
    x = synth.x_gaussian(B, T, m, seed=9, tag="c/x")
    x[:, :, 0] = np.clip(x[:, :, 0], -4, 4) * np.float32(x_scale)
    y0 = np.clip(synth.normal(9, "c/y0", (B, n)), -3, 3) * np.float32(y0_scale)
    args = bd.GruParamsDev.from_numpy(p), dev(x), dev(y0)
    r, names = launched(bd, lambda: bd.deer_gru_eval(*args))
    assert ONE in names and not behind(names) and (kernel is None or m > 64) == projected(names), names
    assert r.status == 0 and r.err <= 1e-4
    want = oracle.gru_seq(p, x, y0, np.float64)
    assert np.max(np.abs(r.y.cpu().numpy() - want)) <= (3e-6 if y0_scale < 1.0 and x_scale == 1.0 else 1e-4)


@pytest.mark.parametrize("n,m,B,T,x_scale,kernel", [
    (9, 3, 10, 300, 1.0, SEG), (12, 17, 3, 401, 1.0, SEG), (16, 8, 4, 501, 1.0, SEG), (24, 16, 16, 6001, 1.0, SEG), (31, 33, 2, 301, 1.0, SEG),
    (32, 5, 2, 301, 1.0, SEG), (40, 7, 4, 301, 1.0, SEG), (48, 1, 2, 201, 1.0, SEG), (24, 4, 3, 401, 3000.0, SEG), (24, 4, 3, 401, 2e4, None)])
def test_two_phase_products_are_at_fp32_level(bd, n, m, B, T, x_scale, kernel):
    """As above, for the two-phase form; n = 16 keeps TF32 products, good to 2^-20."""
    p = synth.gru_params(n, m, seed=10, tag="c/gru")
    x = synth.x_gaussian(B, T, m, seed=10, tag="c/x")
    x[:, :, 0] = np.clip(x[:, :, 0], -4, 4) * np.float32(x_scale)
    y0 = synth.normal(10, "c/y0", (B, n)) * 0.5
    args = bd.GruParamsDev.from_numpy(p), dev(x), dev(y0)
    r, names = launched(bd, lambda: bd.deer_gru_eval(*args))
    assert SEG in names and not behind(names) and (kernel is None) == projected(names), names
    assert r.status == 0 and r.err <= 1e-4
    want = oracle.gru_seq(p, x, y0, np.float64)
    assert np.max(np.abs(r.y.cpu().numpy() - want)) <= (3e-6 if x_scale == 1.0 else 1e-4)


def units(m, kind):
    """A unit per channel: all of them small, all large, or each of its own."""
    return (np.full(m, 1e-6) if kind == "small" else np.full(m, 1e5) if kind == "large" else 10.0 ** np.linspace(-7, 6, m)).astype(np.float32)


@pytest.mark.parametrize("n,m,B,T,kernel", [
    (9, 3, 10, 300, SEG), (24, 8, 3, 401, SEG), (24, 16, 16, 6001, SEG), (32, 5, 2, 301, SEG), (40, 33, 4, 301, SEG),
    (12, 16, 16, 40001, ONE), (16, 5, 16, 15001, ONE), (43, 64, 5, 2003, ONE), (62, 20, 4, 663, ONE),
    (32, 33, 16, 16001, TILE), (32, 5, 16, 8001, TILE), (64, 64, 7, 2801, TILE), (64, 6, 3, 9001, TILE)])
@pytest.mark.parametrize("kind", ["small", "large", "mixed"])
def test_products_do_not_depend_on_the_unit_of_an_input(bd, n, m, B, T, kernel, kind):
    """A normalisation folded into the first layer: x s and W_i / s for x and W_i.  The same bounds as of data of order one: the gates'
    2e-7, less than ten times of it carried, and no other kernel does the work."""
    p = synth.gru_params(n, m, seed=20, tag="c/gru")
    s = units(m, kind)
    p.W_i[:] = p.W_i / s
    x = synth.x_gaussian(B, T, m, seed=20, tag="c/x") * s
    y0 = synth.normal(20, "c/y0", (B, n)) * 0.5
    args = bd.GruParamsDev.from_numpy(p), dev(x), dev(y0)
    r, names = launched(bd, lambda: bd.deer_gru_eval(*args))
    assert kernel in names and not behind(names), names
    assert r.status == 0 and r.err <= 1e-4
    assert np.max(np.abs(r.y.cpu().numpy() - oracle.gru_seq(p, x, y0, np.float64))) <= 3e-6


@pytest.mark.parametrize("n,m,B,T,kernel", [
    (12, 5, 8, 3001, WARP), (17, 16, 16, 700, WARP), (32, 32, 16, 8001, WARP), (48, 2, 16, 500, WARP), (63, 40, 16, 700, WARP),
    (64, 6, 4, 20001, MMA_TILE), (64, 61, 16, 4003, MMA_TILE)])
@pytest.mark.parametrize("kind", ["small", "large", "mixed"])
def test_adjoint_products_do_not_depend_on_the_unit_of_an_input(bd, n, m, B, T, kernel, kind):
    """As above, for the adjoint: 2-norms agree to 1e-6, of dx channel by channel.  (The trajectory that the gradient is taken at is
    given; its gates are evaluated anew.)"""
    p = synth.gru_params(n, m, 21, tag="c/gru")
    s = units(m, kind)
    p.W_i[:] = p.W_i / s
    x = synth.x_gaussian(B, T, m, 21, tag="c/x") * s
    y0 = synth.normal(21, "c/y0", (B, n)) * 0.3
    gy = synth.normal(21, "c/gy", (B, T, n))
    got, want, names, done = gradient(bd, p, x, y0, gy)
    assert kernel in names and done == 1, names
    for k in ("db_i", "db_h", "dy0"):
        assert np.linalg.norm(got[k] - want[k]) <= 1e-6 * np.linalg.norm(want[k]), k
    for c in range(m):
        assert np.linalg.norm(got["dx"][..., c] - want["dx"][..., c]) <= 1e-6 * np.linalg.norm(want["dx"][..., c]), c


@pytest.mark.parametrize("n,m,B,T,kernel", [(24, 4, 3, 401, SEG), (24, 4, 16, 40001, ONE), (32, 32, 16, 6001, TILE)])
@pytest.mark.parametrize("slow", [False, True])
@pytest.mark.parametrize("where", ["x", "y0"])
def test_values_beyond_f16(bd, n, m, B, T, kernel, slow, where):
    """An input that an operand cannot hold: the chains by warps run again with projected inputs, the tiles leave it to the kernels
    without f16 operands.  So is a state of that size, and no other form of the same range is tried, whatever an earlier call has
    left behind (a cell that forgets, or one that was given up because it does not)."""
    p = synth.gru_params(n, m, seed=22, tag="c/gru")
    q = synth.gru_params(n, m, seed=22, tag="c/gru")
    q.b_i[n:2 * n] += np.float32(8.0 if slow else 0.0)
    x = synth.x_gaussian(B, T, m, seed=22, tag="c/x")
    y0 = dev(np.zeros((B, n), np.float32))
    bd.deer_gru_eval(bd.GruParamsDev.from_numpy(q), dev(x), y0)
    start = np.zeros((B, n), np.float32)
    if where == "x":
        x[1, 100] = 1e9 * np.sign(x[1, 100])
    else:
        start[1, 3] = 1e5
    r, names = launched(bd, lambda: bd.deer_gru_eval(bd.GruParamsDev.from_numpy(p), dev(x), dev(start), max_iter=20))
    assert names & {SEG, ONE, TILE} == {kernel} and behind(names) == (where == "y0" or kernel == TILE), names
    if where == "x":                   # (from such a start the iteration does not converge in any form)
        assert r.status == 0
        assert np.max(np.abs(r.y.cpu().numpy() - oracle.gru_seq(p, x, start, np.float32))) <= 1e-4


@pytest.mark.parametrize("n,m,B,T,kernel", [(4, 3, 16, 50003, LANE), (8, 8, 16, 30001, LANE), (32, 33, 16, 16001, TILE), (64, 6, 3, 9001, TILE)])
@pytest.mark.parametrize("tol", [1e-6, 1e-7])
def test_a_tolerance_below_what_a_boundary_can_show(bd, n, m, B, T, kernel, tol):
    """Where a boundary's mismatch is the rounding of two states the tolerance decides whether that is enough, here not: the result is
    no further off than that of the kernels that multiply the Jacobians out, but for the difference of two roundings carried on."""
    p = synth.gru_params(n, m, seed=23, tag="c/gru")
    p.b_i[n:2 * n] += np.float32(1.5)
    x = synth.x_gaussian(B, T, m, seed=23, tag="c/x")
    y0 = synth.normal(23, "c/y0", (B, n)) * 0.5
    args = bd.GruParamsDev.from_numpy(p), dev(x), dev(y0)
    r, names = launched(bd, lambda: bd.deer_gru_eval(*args, tol=tol))
    other = bd.deer_gru_eval(*args, tol=tol, flags=bd.DEER_FLAG_MATERIALIZE)
    assert kernel in names and behind(names), names
    assert r.status == 0 and r.err <= tol or r.status == bd.DEER_NOT_CONVERGED      # (updates of 1e-7 are the rounding of a state near one: they may not end)
    want = oracle.gru_seq(p, x, y0, np.float64)
    off = [np.max(np.abs(q.y.cpu().numpy() - want)) for q in (r, other)]
    assert off[0] <= 1.5 * off[1] + 2.4e-7, off


def test_updates_of_some_hundred_stay_with_the_chains(bd):
    """A start far from anything that a gate gives: updates of up to 140 on the way, and the chains' f16 operands hold them.  (Much
    larger ones come of iterations that do not converge in any form.)"""
    n, m, B, T = 9, 3, 10, 300
    p = synth.gru_params(n, m, seed=24, tag="c/gru")
    x = synth.x_gaussian(B, T, m, seed=24, tag="c/x")
    y0 = np.clip(synth.normal(24, "c/y0", (B, n)), -3, 3) * np.float32(30.0)
    r, names = launched(bd, lambda: bd.deer_gru_eval(bd.GruParamsDev.from_numpy(p), dev(x), dev(y0)))
    assert SEG in names and not behind(names), names
    assert r.status == 0 and r.err <= 1e-4 and max(r.err_trace[:r.iters]) > 64
