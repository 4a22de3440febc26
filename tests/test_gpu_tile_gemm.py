"""The dense products of a multi-head unit (projection, dx, the weights' sums): tiles of 128 x 256, stages of 32, two of them."""
import numpy as np
import pytest
import torch

import oracle
from paper_2309_12252_b200 import binding as bd
from paper_2309_12252_b200 import synth

pytestmark = pytest.mark.gpu


# one column and one stage; sizes that are no multiple of 4 (n, m); a tile's edge in positions (128, 129), inputs (255, 257) and stacked
# gates (16 heads of 24: 384 = 3 tiles; 11 of 12: a head across two tiles); strides longer than the sequence; one position; more than a
# wave of tiles of 128 columns, rows of C on and off 32 bytes
@pytest.mark.parametrize("H,n,m,B,T,strides", [
    (1, 1, 1, 1, 1, [1]), (2, 4, 8, 1, 128, [1, 2]), (3, 7, 5, 3, 43, [1, 4, 64]), (11, 4, 255, 1, 129, [1, 2, 4, 8, 1, 2, 4, 8, 1, 2, 4]),
    (16, 8, 257, 2, 97, [1, 2, 4, 8] * 4), (2, 64, 32, 2, 33, [1, 3]), (5, 30, 36, 4, 160, [1, 2, 3, 4, 5]), (6, 16, 256, 16, 300, [1, 2, 4, 8, 16, 32]),
    (3, 6, 257, 16, 1201, [1, 2, 64]), (2, 16, 264, 16, 1201, [1, 4]),
])
def test_multihead_gradients_against_the_oracle(H, n, m, B, T, strides):
    hp = [synth.gru_params(n, m, seed=31 + h, tag="t/gru") for h in range(H)]
    heads = [bd.GruParamsDev.from_numpy(p) for p in hp]
    x = synth.x_gaussian(B, T, m, seed=31, tag="t/x")
    y0 = synth.normal(31, "t/y0", (B, H, n)) * np.float32(0.5)
    gy = synth.normal(31, "t/gy", (B, T, H, n))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    y, _, status = bd.deer_gru_multihead_eval(heads, strides, dev(x), dev(y0), tol=1e-6)
    assert status == 0
    got = bd.deer_gru_multihead_vjp(heads, strides, dev(x), dev(y0), y, dev(gy))
    yn = y.cpu().numpy()
    dx, dy0, want = np.zeros((B, T, m)), np.zeros((B, H, n)), []
    for h, s in enumerate(strides):
        acc = None
        for ph in range(min(s, T)):
            part = [np.ascontiguousarray(a) for a in (x[:, ph::s], y0[:, h], yn[:, ph::s, h], gy[:, ph::s, h])]
            seq = oracle.gru_seq(hp[h], part[0], part[1], np.float32)
            assert np.max(np.abs(seq - part[2])) <= 1e-5          # fp32 trajectories of another order of summation
            w = oracle.gru_bptt(hp[h], part[0], part[1], part[2].astype(np.float64), part[3], np.float64)
            dx[:, ph::s] += w["dx"]
            dy0[:, h] += w["dy0"]
            acc = {k: (acc[k] + w[k] if acc else w[k].copy()) for k in ("dW_i", "dW_h", "db_i", "db_h")}
        want.append(acc)
    near = lambda a, b: np.linalg.norm(a.cpu().numpy() - b) <= 8e-6 * np.linalg.norm(b)      # adjoint 4e-6, gates and sums 1e-6
    for k in ("dW_i", "dW_h", "db_i", "db_h"):
        for h in range(H):
            assert near(got[k][h], want[h][k]), (k, h)
    assert near(got["dx"], dx) and near(got["dy0"], dy0)


@pytest.mark.parametrize("H,n,m,N,one_sign", [
    (32, 64, 33, 32768, False), (32, 64, 33, 32768, True), (64, 64, 256, 8192, False), (64, 40, 7, 9600, True), (3, 5, 6, 150016, False),
    (1, 64, 300, 65600, True)])
def test_sums_over_many_positions(H, n, m, N, one_sign):
    """The weights' sums in as few slices as the unit's size leaves, over many stages: every head's stride is the length of the
    sequences, so that each position is a sequence of its own, and the gradients are sums over N positions in 64 bits."""
    T = 8
    g = torch.Generator(device="cuda").manual_seed(41)
    rand = lambda *s: torch.rand(s, generator=g, device="cuda")
    heads = []
    for h in range(H):
        W = [(rand(3 * n, k) * 2 - 1) / n ** 0.5 for k in (m, n)]
        heads.append(bd.GruParamsDev(n, m, *W, (rand(3 * n) - 0.5) * 0.5, (rand(3 * n) - 0.5) * 0.5))
    x = rand(N // T, T, m) - (0.0 if one_sign else 0.5)
    y0 = rand(N // T, H, n) - (0.0 if one_sign else 0.5)
    gy = rand(N // T, T, H, n) - (0.0 if one_sign else 0.5)
    got = bd.deer_gru_multihead_vjp(heads, [T] * H, x, y0, torch.zeros_like(gy), gy)
    X = x.view(N, m).double()
    for h in range(0, H, 7):
        p = heads[h]
        W_i, W_h, b_i, b_h = (t.double() for t in (p.W_i, p.W_h, p.b_i, p.b_h))
        hp, lam = y0[:, h].double().repeat_interleave(T, 0), gy[:, :, h].reshape(N, n).double()
        u, q = X @ W_i.T + b_i, hp @ W_h.T + b_h
        r, z = torch.sigmoid(u[:, :n] + q[:, :n]), torch.sigmoid(u[:, n:2 * n] + q[:, n:2 * n])
        c = torch.tanh(u[:, 2 * n:] + r * q[:, 2 * n:])
        dn = lam * (1 - z) * (1 - c * c)
        dr, dz = dn * q[:, 2 * n:] * r * (1 - r), lam * (hp - c) * z * (1 - z)
        gi, gh = torch.cat([dr, dz, dn], 1), torch.cat([dr, dz, dn * r], 1)
        want = dict(dW_i=gi.T @ X, dW_h=gh.T @ hp, db_i=gi.sum(0), db_h=gh.sum(0))
        for k in want:
            # 128 additions between two flushes, each cutting half of 2^-23 of what is there, on average half of the whole: 3.8e-6;
            # the gates 1e-6 (of the terms, which cancel where they have both signs: the biases' sums are held to the terms there)
            size = want[k].norm() if one_sign or k[1] == "W" else max(want[k].norm(), gi.norm())
            assert (got[k][h].double() - want[k]).norm() <= 5e-6 * size, (k, h)


def test_inputs_masked_with_the_lowest_value():
    """Masked steps hold the type's lowest value in one channel: the projections are finite there, the gates closed or open, and the
    gradients what the other steps give."""
    H, n, m, B, T = 3, 8, 20, 4, 60
    hp = [synth.gru_params(n, m, seed=51 + h, tag="t/gru") for h in range(H)]
    heads = [bd.GruParamsDev.from_numpy(p) for p in hp]
    x = synth.x_gaussian(B, T, m, seed=51, tag="t/x")
    x[1, 7, 3], x[2, 30:33, 0] = np.finfo(np.float32).min, np.finfo(np.float32).min
    gy = synth.normal(51, "t/gy", (B, T, H, n))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    xd, y0 = dev(x), torch.zeros((B, H, n), device="cuda")
    y, _, status = bd.deer_gru_multihead_eval(heads, [1] * H, xd, y0, tol=1e-6)
    assert status == 0
    got = bd.deer_gru_multihead_vjp(heads, [1] * H, xd, y0, y, dev(gy))
    dx = np.zeros((B, T, m))
    for h in range(H):
        zero, yn, g = np.zeros((B, n), np.float32), np.ascontiguousarray(y[:, :, h].cpu().numpy()), np.ascontiguousarray(gy[:, :, h])
        with np.errstate(over="ignore"):
            assert np.max(np.abs(oracle.gru_seq(hp[h], x, zero, np.float32) - yn)) <= 1e-5
            want = oracle.gru_bptt(hp[h], x, zero, yn.astype(np.float64), g, np.float64)
        for k in ("dW_i", "dW_h", "db_i", "db_h"):
            assert np.linalg.norm(got[k][h].cpu().numpy() - want[k]) <= 8e-6 * np.linalg.norm(want[k]), (k, h)
        dx += want["dx"]
    assert np.linalg.norm(got["dx"].cpu().numpy() - dx) <= 8e-6 * np.linalg.norm(dx)


# products of one or two stages (no wait but those behind the last one), of several
@pytest.mark.parametrize("H,n,m,B,T", [(2, 8, 5, 1, 32), (6, 16, 100, 16, 300)])
def test_expired_waits_are_reported(H, n, m, B, T):
    """The waits of one dense product run out at a time, and nothing else's: the call says so, and the next one is right."""
    heads, strides = [bd.GruParamsDev.from_numpy(synth.gru_params(n, m, seed=61 + h, tag="t/gru")) for h in range(H)], [1, 2, 4, 1, 2, 4][:H]
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    x, y0, gy = dev(synth.x_gaussian(B, T, m, seed=61, tag="t/x")), torch.zeros((B, H, n), device="cuda"), dev(synth.normal(61, "t/gy", (B, T, H, n)))
    ws = bd.alloc_multihead_workspace(heads, strides, B, T, x.device)
    y = bd.deer_gru_multihead_eval(heads, strides, x, y0)[0]
    want = bd.deer_gru_multihead_vjp(heads, strides, x, y0, y, gy)
    expired = lambda call: pytest.raises(bd.DeerError, call).value.status == bd.DEER_ERR_DEVICE_TIMEOUT
    assert expired(lambda: bd.deer_gru_multihead_eval(heads, strides, x, y0, ws=ws, flags=bd.DEER_FLAG_EXPIRE_PRODUCT_WAITS))
    again, _, status = bd.deer_gru_multihead_eval(heads, strides, x, y0, ws=ws)
    assert status == bd.DEER_OK and torch.equal(again, y)
    for k in range(4):
        assert expired(lambda: bd.deer_gru_multihead_vjp(heads, strides, x, y0, y, gy, ws=ws, flags=bd.DEER_FLAG_EXPIRE_PRODUCT_WAITS << k)), k
        got = bd.deer_gru_multihead_vjp(heads, strides, x, y0, y, gy, ws=ws)
        for name, v in want.items():
            assert all(torch.equal(a, b) for a, b in zip(got[name], v)), name
