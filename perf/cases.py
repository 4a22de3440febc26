"""What a user of this library has it do, as measurable cases: evaluations of GRUs over whole sequences, their gradients,
training steps, the call with host buffers, the multi-head unit and the stand-alone linear recurrence.

A case is a dict of plain values.  ``kind`` names the entry point:

``eval``        deer_gru_eval, device buffers             (n, m, B, T, x, memory)
``host``        deer_gru_eval_host, pinned host buffers   (n, m, B, T)
``grad``        deer_gru_vjp at an evaluated trajectory   (n, m, B, T)
``classifier``  deer_gru_classifier_step                  (n, m, B, T, classes)
``multihead``   deer_gru_multihead_eval, then its _vjp    (heads, n, m, B, T)
``scan``        deer_linrec_scan                          (n, B, T, reverse)

Everything is fp32, as the library's interface is.  GRU weights are those of an untrained cell, U(-1/sqrt n, 1/sqrt n);
``memory`` > 0 adds log U(1, memory) to the update gate's bias, the usual initialisation of a cell that has to remember for
up to that many steps.  ``x`` is white noise (``noise``), noisy sinusoids (``wave``) or z-normalised random walks (``walk``).
"""
import math

import torch

from paper_2309_12252_b200 import binding as deer

TOL = 1e-4              # the evaluation's stopping tolerance: the library's default
MAX_STRIDE_EXP = 8      # strides of a multi-head unit's heads: 2^0 ... 2^7, in turn


def listed():
    return [
        # one short sequence of a small cell: all latency and launches
        dict(name="eval n4 short", kind="eval", n=4, m=2, B=1, T=1000, x="noise", memory=0),
        # a batch of ordinary length, small state
        dict(name="eval n8 wave", kind="eval", n=8, m=4, B=16, T=10000, x="wave", memory=0),
        # the longest sequences: a scalar state over a million steps
        dict(name="eval n1 million", kind="eval", n=1, m=1, B=16, T=1000000, x="noise", memory=0),
        # a wide state over long sequences: the benchmark's headline size
        dict(name="eval n32 long", kind="eval", n=32, m=32, B=16, T=100000, x="noise", memory=0),
        # sizes that are no powers of two, ragged everywhere
        dict(name="eval n24 ragged", kind="eval", n=24, m=10, B=5, T=4001, x="walk", memory=0),
        # a cell initialised to remember for long: Jacobian products that hardly decay
        dict(name="eval n16 memory", kind="eval", n=16, m=8, B=8, T=20000, x="noise", memory=1000),
        # the headline size from and to host memory
        dict(name="host n32 long", kind="host", n=32, m=32, B=16, T=100000),
        # gradients through a small and through a wide evaluation
        dict(name="grad n8", kind="grad", n=8, m=4, B=16, T=10000),
        dict(name="grad n32 long", kind="grad", n=32, m=32, B=16, T=100000),
        # a whole training step of the two-layer long-series classifier
        dict(name="classifier n64", kind="classifier", n=64, m=6, B=32, T=17984, classes=5),
        # forward and backward of the multi-head unit of the sequential-image model
        dict(name="multihead 32x8", kind="multihead", heads=32, n=8, m=256, B=32, T=1024),
        # the linear recurrence by itself, on Jacobians larger than L2
        dict(name="scan n8", kind="scan", n=8, B=16, T=200000, reverse=False),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _split(rng, positions, max_B, min_T):
    """B sequences of T steps with about that many positions in all."""
    B = max(1, min(int(_log(rng, 1, max_B + 1)), int(positions / min_T)))
    return B, max(min_T, int(positions / B))


def _width(rng):
    """A state size: half of them the powers of two that cells are usually given, half anything up to 64."""
    return rng.choice([1, 2, 4, 8, 16, 32, 64]) if rng.random() < 0.5 else rng.randint(1, 64)


def _most(n):
    """Positions at most: as many state-by-state entries as the wide listed evaluation has; fewer where n is no power of two."""
    most = 1.6e6 * (32.0 / n) ** 2
    return min(1.6e7, most) if n & (n - 1) == 0 else min(1e6, 0.04 * most)


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "eval", "host", "grad", "grad", "classifier", "multihead", "scan"])
    if kind in ("eval", "grad"):
        n = _width(rng)
        B, T = _split(rng, _log(rng, 1e3, _most(n)), 64, 64)
        m = int(_log(rng, 1, 65))
        m = min(m, max(1, int(5.2e7 / (B * T))))
        c = dict(kind=kind, n=n, m=m, B=B, T=T)
        if kind == "eval":
            c.update(x=rng.choice(["noise", "wave", "walk"]), memory=rng.choice([0, 0, 0, 0, 1000]))
        return c
    if kind == "host":
        n = rng.choice([4, 8, 16, 32])
        B, T = _split(rng, _log(rng, 2e4, 1.6e6), 64, 64)
        return dict(kind=kind, n=n, m=int(_log(rng, 1, 33)), B=B, T=T)
    if kind == "classifier":
        B, T = _split(rng, _log(rng, 1e4, 5e5), 32, 128)
        return dict(kind=kind, n=rng.choice([8, 16, 32, 64]), m=rng.randint(1, 12), B=B, T=T, classes=rng.randint(2, 10))
    if kind == "multihead":
        return dict(kind=kind, heads=rng.randint(2, 32), n=rng.choice([4, 8, 16]), m=int(_log(rng, 8, 257)), B=rng.randint(1, 32),
                    T=int(_log(rng, 128, 1025)))
    n = rng.choice([1, 2, 4, 8, 16, 32, 64])
    B, T = _split(rng, _log(rng, 1e4, min(1.6e7, 2.5e8 / n ** 2)), 64, 64)
    return dict(kind=kind, n=n, B=B, T=T, reverse=rng.random() < 0.5)


# ---------------------------------------------------------------- inputs
def _uniform(g, shape, a):
    return (torch.rand(shape, generator=g, device="cuda") * 2 - 1) * a


def _params(g, n, m, memory=0):
    a = 1.0 / math.sqrt(n)
    p = deer.GruParamsDev(n, m, _uniform(g, (3 * n, m), a), _uniform(g, (3 * n, n), a), _uniform(g, (3 * n,), a),
                          _uniform(g, (3 * n,), a))
    if memory:
        p.b_i[n:2 * n] += torch.log(1 + (memory - 1) * torch.rand((n,), generator=g, device="cuda"))
    return p


def _x(g, B, T, m, how="noise"):
    if how == "wave":
        w = 0.001 + 0.099 * torch.rand((B, 1, m), generator=g, device="cuda")
        phase = 2 * math.pi * torch.rand((B, 1, m), generator=g, device="cuda")
        x = torch.arange(T, device="cuda", dtype=torch.float32).reshape(1, T, 1) * w
        x = x.add_(phase).sin_()
        return x.add_(torch.randn((B, T, m), generator=g, device="cuda"), alpha=0.1)
    x = torch.randn((B, T, m), generator=g, device="cuda")
    if how == "walk":
        x = torch.cumsum(x.double(), dim=1)
        x = ((x - x.mean(dim=1, keepdim=True)) / x.std(dim=1, keepdim=True, unbiased=False)).float()
    return x


def _jacobians(g, n, B, T):
    """Jacobians of an untrained GRU along a guess: diag(z) + diag(k_r) W_hr + diag(a_z) W_hz + diag(k_n) W_hn."""
    p = _params(g, n, n)
    W_r, W_z, W_n = p.W_h.split(n)
    J = torch.empty((B, T, n, n), device="cuda")
    for b in range(B):                                                  # one sequence at a time: the matrices are large
        u = torch.randn((T, n), generator=g, device="cuda") @ p.W_i.T + p.b_i
        h = torch.tanh(torch.randn((T, n), generator=g, device="cuda") * 0.5)
        q = h @ p.W_h.T + p.b_h
        r, z = torch.sigmoid(u[:, :n] + q[:, :n]), torch.sigmoid(u[:, n:2 * n] + q[:, n:2 * n])
        c = torch.tanh(u[:, 2 * n:] + r * q[:, 2 * n:])
        k = (1 - z) * (1 - c * c)
        Jb = J[b]
        torch.mul((k * r).unsqueeze(2), W_n, out=Jb)
        Jb.addcmul_((k * q[:, 2 * n:] * r * (1 - r)).unsqueeze(2), W_r)
        Jb.addcmul_(((h - c) * z * (1 - z)).unsqueeze(2), W_z)
        Jb.diagonal(dim1=1, dim2=2).add_(z)
    return J


def prepare(case, seed):
    c = dict(case)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind, n, B, T = c["kind"], c["n"], c["B"], c["T"]
    s = dict(kind=kind)
    if kind == "scan":
        s.update(J=_jacobians(g, n, B, T), b=torch.randn((B, T, n), generator=g, device="cuda"), reverse=bool(c["reverse"]),
                 y0=torch.randn((B, n), generator=g, device="cuda"), y=torch.empty((B, T, n), device="cuda"),
                 ws=deer.alloc_workspace(deer.DEER_OP_SCAN, B, T, n))
        return s
    m = c["m"]
    if kind == "classifier":
        a = 1.0 / math.sqrt(n)
        s.update(l1=_params(g, n, m), l2=_params(g, n, n), W_o=_uniform(g, (c["classes"], n), a), b_o=_uniform(g, (c["classes"],), a),
                 x=_x(g, B, T, m, "walk"),
                 labels=torch.randint(0, c["classes"], (B,), generator=g, device="cuda", dtype=torch.int32),
                 ws=deer.alloc_workspace(deer.DEER_OP_CLASSIFIER, B, T, n, m))
        return s
    if kind == "multihead":
        heads = [_params(g, n, m) for _ in range(c["heads"])]
        strides = [2 ** (h % MAX_STRIDE_EXP) for h in range(c["heads"])]
        s.update(heads=heads, strides=strides, x=_x(g, B, T, m), y0=torch.zeros((B, c["heads"], n), device="cuda"),
                 gy=torch.randn((B, T, c["heads"], n), generator=g, device="cuda"),
                 y=torch.empty((B, T, c["heads"], n), device="cuda"),
                 ws=deer.alloc_multihead_workspace(heads, strides, B, T))
        return s
    p = _params(g, n, m, c.get("memory", 0))
    x = _x(g, B, T, m, c.get("x", "noise"))
    y0 = torch.zeros((B, n), device="cuda")
    y = torch.empty((B, T, n), device="cuda")
    s.update(p=p, x=x, y0=y0, y=y)
    if kind == "grad":
        deer.deer_gru_eval(p, x, y0, tol=TOL, y=y)
        s.update(gy=torch.randn((B, T, n), generator=g, device="cuda"), ws=deer.alloc_workspace(deer.DEER_OP_VJP, B, T, n, m))
        return s
    s["ws"] = deer.alloc_workspace(deer.DEER_OP_EVAL, B, T, n, m)
    if kind == "host":
        s["x_host"] = torch.empty((B, T, m), pin_memory=True).copy_(x)
        s["y_host"] = torch.empty((B, T, n), pin_memory=True)
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    kind = s["kind"]
    if kind == "eval":
        return deer.deer_gru_eval(s["p"], s["x"], s["y0"], tol=TOL, y=s["y"], ws=s["ws"]).y
    if kind == "host":
        deer.deer_gru_eval_host(s["p"], s["x_host"], s["y0"], s["y_host"], s["x"], s["y"], s["ws"], tol=TOL)
        return s["y_host"]
    if kind == "grad":
        return deer.deer_gru_vjp(s["p"], s["x"], s["y0"], s["y"], s["gy"], ws=s["ws"])
    if kind == "classifier":
        r = deer.deer_gru_classifier_step(s["l1"], s["l2"], s["W_o"], s["b_o"], s["x"], s["labels"], tol=TOL, ws=s["ws"])
        return {k: r[k] for k in ("loss", "g1", "g2", "dW_o", "db_o")}
    if kind == "multihead":
        y, _, _ = deer.deer_gru_multihead_eval(s["heads"], s["strides"], s["x"], s["y0"], tol=TOL, y=s["y"], ws=s["ws"])
        g = deer.deer_gru_multihead_vjp(s["heads"], s["strides"], s["x"], s["y0"], y, s["gy"], ws=s["ws"])
        # the parameters' gradients as the one flat vector that an optimiser or a clipping step takes
        flat = torch.cat([t.reshape(-1) for k in ("dW_i", "dW_h", "db_i", "db_h") for t in g[k]])
        return dict(y=y, grads=flat, dx=g["dx"], dy0=g["dy0"])
    return deer.deer_linrec_scan(s["J"], s["b"], s["y0"], reverse=s["reverse"], y=s["y"], ws=s["ws"])


def work(case):
    c = dict(case)
    kind, n, N = c["kind"], c["n"], c["B"] * c["T"]
    if kind == "scan":
        return dict(bytes=4 * N * (n * n + 2 * n), flops=2 * N * n * n)
    m = c["m"]
    cell = 6 * n * (n + m)                          # the gates' products at one position
    weights = 4 * 3 * n * (n + m + 2)
    if kind in ("eval", "host"):
        return dict(bytes=4 * N * (m + n) + weights, flops=N * cell)
    if kind == "grad":                              # gates, adjoint step, parameter gradients, dx
        return dict(bytes=4 * N * (2 * m + 2 * n) + 2 * weights, flops=N * (2 * cell + 6 * n * n + 6 * n * m))
    if kind == "classifier":                        # two layers forward and backward; dx of the second layer only
        f = sum(N * (3 * 6 * n * (n + k) + 6 * n * n) for k in (m, n)) + N * 6 * n * n
        return dict(bytes=4 * N * (m + 2 * n), flops=f)
    H = c["heads"]
    return dict(bytes=4 * N * (2 * m + 3 * H * n) + 2 * H * weights, flops=N * H * (3 * cell + 6 * n * n + 6 * n * m))


def tolerance(case):
    kind = case["kind"]
    if kind in ("eval", "host"):
        return {"rel": 5e-5, "max": 1e-3}           # an iteration that stops at updates of 1e-4
    if kind in ("classifier", "multihead"):
        return {"rel": 1e-4, "max": 4e-3}           # gradients at such a trajectory
    return {"rel": 2e-5, "max": 8e-4}               # one solve in 32 bits
