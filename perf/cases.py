"""The work that this solver's speed is judged on, through its public entry points.

Each case is one call (or the few calls) that a program makes per unit of work: a whole solve
(factor and refine), a refinement with a factor that the program keeps, a conjugate-gradient solve,
a batched solve, a training step of the learned preconditioner.  The inputs are made on the GPU from
the seed.  Matrices are those of the benchmark and the tests: prescribed spectrum, shifted Gram,
exponential covariance, the model covariance 1/|i-j|^d, Matern-3/2.
"""
import math
import random

import torch

import paper_1405_4644_gb300 as spd
from paper_1405_4644_gb300 import learned

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # one small system, one right-hand side, all defaults: launches and latency
        {"name": "plain_1024", "kind": "solve", "matrix": "gram", "n": 1024, "m": 1, "prec": "auto", "resid": "fp64"},
        # a mid-sized well-conditioned system of odd order with a few right-hand sides, 16-bit factor
        {"name": "ragged_2999_bf16", "kind": "solve", "matrix": "spectrum", "kappa": 8.0, "n": 2999, "m": 5,
         "prec": "bf16", "resid": "auto"},
        # a program that keeps its factor and solves for new right-hand sides
        {"name": "refine_8191", "kind": "refine", "matrix": "spectrum", "kappa": 1e3, "n": 8191, "m": 32,
         "prec": "fp32", "resid": "auto"},
        # the benchmark's systems: AUTO keeps an FP16 factor for the first and takes FP32 for the second
        {"name": "bench_16384_k2", "kind": "solve", "matrix": "spectrum", "kappa": 1e2, "n": 16384, "m": 16,
         "prec": "auto", "resid": "tc"},
        {"name": "bench_16384_k4", "kind": "solve", "matrix": "spectrum", "kappa": 1e4, "n": 16384, "m": 16,
         "prec": "auto", "resid": "tc"},
        # the largest: the exponential covariance of 32768 points
        {"name": "cov_32768", "kind": "solve", "matrix": "cov", "n": 32768, "m": 8, "prec": "fp32", "resid": "auto"},
        # conjugate gradients on the model covariance: bound by the matrix at one right-hand side, a
        # contraction at 32, and the banded inner matrix, where every step is a few launches
        {"name": "cg_16384_1", "kind": "cg", "n": 16384, "m": 1, "d": 1, "band": -1},
        {"name": "cg_16384_32", "kind": "cg", "n": 16384, "m": 32, "d": 2, "band": -1},
        {"name": "cg_band_16384", "kind": "cg", "n": 16384, "m": 1, "d": 4, "band": 16},
        # thousands of systems of uneven order in one launch, and a smaller batch by Jacobi-PCG
        {"name": "batch_4096", "kind": "batch", "method": "chol_ir", "count": 4096, "nmin": 32, "nmax": 512,
         "prec": "fp32"},
        {"name": "batch_pcg_512", "kind": "batch", "method": "pcg_jacobi", "count": 512, "nmin": 32, "nmax": 256,
         "prec": "fp32"},
        # one training step of the learned preconditioner: features, probe loss and its gradient
        {"name": "learned_4096", "kind": "learned", "n": 4096, "p": 8, "hidden": 256, "bf16": True, "ell": 0.1,
         "nugget": 0.05},
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "refine", "cg", "band", "batch", "pcg", "learned"])
    if kind == "solve":
        prec = rng.choice(["auto", "auto", "fp32", "fp32", "fp16", "tf32", "bf16"])
        top = {"auto": 1e5, "fp32": 1e5, "fp16": 1e2, "tf32": 1e2, "bf16": 1e1}[prec]
        n, m = _log(rng, 128, 16384), _log(rng, 1, 64)
        return {"kind": "solve", "matrix": "spectrum", "kappa": round(10 ** rng.uniform(0.6, math.log10(top)), 2),
                "n": n, "m": m, "prec": prec, "resid": "fp64" if n <= 3000 and rng.random() < 0.5 else "auto"}
    if kind == "refine":
        return {"kind": "refine", "matrix": "spectrum", "kappa": round(10 ** rng.uniform(1, 4.5), 2),
                "n": _log(rng, 1024, 12288), "m": _log(rng, 1, 64), "prec": "fp32", "resid": "auto"}
    if kind == "cg":
        return {"kind": "cg", "n": _log(rng, 512, 16384), "m": _log(rng, 1, 64), "d": rng.choice([1, 2, 4]),
                "band": -1}
    if kind == "band":
        return {"kind": "cg", "n": _log(rng, 1024, 16384), "m": _log(rng, 1, 32), "d": rng.choice([2, 4]),
                "band": rng.randint(4, 32)}
    if kind == "batch":
        nmax = rng.randint(48, 512)
        return {"kind": "batch", "method": "chol_ir", "count": _log(rng, 16, 4096), "nmin": rng.randint(1, 32),
                "nmax": nmax, "prec": rng.choice(["fp32", "fp32", "fp16", "bf16"])}
    if kind == "pcg":
        return {"kind": "batch", "method": "pcg_jacobi", "count": _log(rng, 16, 1024), "nmin": rng.randint(1, 32),
                "nmax": rng.randint(48, 400), "prec": "fp32"}
    return {"kind": "learned", "n": _log(rng, 512, 4096), "p": rng.randint(1, 8), "hidden": rng.choice([64, 128, 256]),
            "bf16": rng.random() < 0.5, "ell": round(rng.uniform(0.05, 0.2), 3),
            "nugget": round(10 ** rng.uniform(-2, -1), 4)}


# ---- inputs ---------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _sym(A):
    """The symmetric part, in row blocks of A itself (no second matrix for the large orders)."""
    n = A.shape[0]
    for i in range(0, n, 4096):
        for j in range(0, i + 1, 4096):
            P, Q = A[i:i + 4096, j:j + 4096], A[j:j + 4096, i:i + 4096]
            S = 0.5 * (P + Q.T)
            P.copy_(S)
            Q.copy_(S.T)
    return A


def _matrix(c, g):
    n = c["n"]
    kind = c.get("matrix", "model")
    if kind == "gram":  # G G^T / n + 0.1 I
        G = torch.randn(n, n, dtype=F64, device=DEV, generator=g)
        A = _sym(G @ G.T / n)
        A.diagonal().add_(0.1)
        return A
    if kind == "spectrum":  # Q diag(lambda) Q^T, Q = 32 Householder reflections, lambda log-spaced in [1, kappa]
        k = min(32, n)
        V = torch.randn(n, k, dtype=F64, device=DEV, generator=g)
        V /= torch.linalg.norm(V, dim=0)
        lam = torch.logspace(0.0, math.log10(c["kappa"]), n, dtype=F64, device=DEV)
        VV = (V.T @ V).cpu()
        T = torch.zeros(k, k, dtype=F64)
        for j in range(k):  # Q = I - V T V^T
            T[j, j] = 2.0
            if j:
                T[:j, j] = -2.0 * (T[:j, :j] @ VV[:j, j])
        T = T.to(DEV)
        W = lam[:, None] * V
        # A = Lam - V T W^T - W T^T V^T + V (T V^T W T^T) V^T
        A = torch.cat([V @ (T @ (V.T @ W) @ T.T) - W @ T.T, -V @ T], 1) @ torch.cat([V, W], 1).T
        A.diagonal().add_(lam)
        return _sym(A)
    if kind == "cov":  # exp(-|p_i - p_j| / 0.1) + 1e-3 I over points of the unit cube
        P = torch.rand(n, 3, dtype=F64, device=DEV, generator=g)
        A = torch.empty(n, n, dtype=F64, device=DEV)
        for r in range(0, n, 2048):
            d = torch.cdist(P[r:r + 2048], P, compute_mode="donot_use_mm_for_euclid_dist")
            torch.exp(d.mul_(-10.0), out=A[r:r + 2048])
        _sym(A)
        A.diagonal().add_(1e-3)
        return A
    # 1 / |i - j|^d, diagonal 1 + sqrt(i)
    i = torch.arange(n, dtype=F64, device=DEV)
    t = 1.0 / torch.clamp(i, min=1.0) ** c["d"]
    A = t[(i[:, None] - i[None, :]).abs_().long()]
    A.diagonal().copy_(1.0 + torch.sqrt(i + 1.0))
    return A


def _system(c, seed):
    g = _gen(seed)
    A = _matrix(c, g)
    if c["kind"] == "cg":  # right-hand sides U[0, 1]
        B = torch.rand(c["m"], c["n"], dtype=F64, device=DEV, generator=g).t()
    else:
        B = torch.randn(c["m"], c["n"], dtype=F64, device=DEV, generator=g).t()
    return A, B


def _batch_sizes(c):
    r = random.Random("%d %d %d" % (c["count"], c["nmin"], c["nmax"]))
    return [r.randint(c["nmin"], c["nmax"]) for _ in range(c["count"])]


def _batch_systems(c, seed):
    """(sizes, A_i = G G^T / n_i + 0.05 I, one flat right-hand side, offsets); systems of one order lie together."""
    g = _gen(seed)
    sizes = _batch_sizes(c)
    As = [None] * len(sizes)
    by = {}
    for i, n in enumerate(sizes):
        by.setdefault(n, []).append(i)
    groups = []
    for n, idx in sorted(by.items()):
        G = torch.randn(len(idx), n, n, dtype=F64, device=DEV, generator=g)
        A = torch.bmm(G, G.transpose(1, 2)).div_(n)
        A = 0.5 * (A + A.transpose(1, 2))
        A.diagonal(dim1=1, dim2=2).add_(0.05)
        for k, i in enumerate(idx):
            As[i] = A[k]
        groups.append((n, idx, A))
    off = [0]
    for n in sizes:
        off.append(off[-1] + n)
    b = torch.randn(off[-1], dtype=F64, device=DEV, generator=g)
    return sizes, As, b, off, groups


def _learned_inputs(c, seed):
    """A Matern-3/2 covariance over points of the unit square, probes, the supervised target, and a network's weights."""
    g = _gen(seed)
    n, H = c["n"], c["hidden"]
    pts = torch.rand(n, 2, dtype=F64, device=DEV, generator=g)
    s = math.sqrt(3.0) / c["ell"] * torch.cdist(pts, pts, compute_mode="donot_use_mm_for_euclid_dist")
    A = _sym((1.0 + s) * torch.exp(-s))
    A.diagonal().add_(c["nugget"])
    Z = torch.randn(c["p"], n, dtype=F64, device=DEV, generator=g).t()
    T = torch.cholesky_solve(Z[:, :1], torch.linalg.cholesky(A)).reshape(n)
    parts = []
    for rows, cols, scale in ((H, 16, 0.25), (H, H, 1.0 / math.sqrt(H)), (33, H, 0.5 / math.sqrt(H))):
        parts.append((torch.rand(rows * cols, device=DEV, generator=g) * 2 - 1) * scale)
        parts.append(0.1 * torch.randn(rows, device=DEV, generator=g))
    parts[-1][0] = 0.54  # softplus(0.54) is about 1: the diagonal of a scaled matrix
    return A, pts, Z, T.contiguous(), torch.cat(parts).float().contiguous()


# ---- states and passes ------------------------------------------------------------------------------------
_handle = None


def _h():
    """The handle that a program keeps for all its calls."""
    global _handle
    if _handle is None:
        _handle = spd.spd_create(torch.cuda.current_stream())
    return _handle


def _ok(st):
    if st != spd.SPD_OK:
        raise RuntimeError("status %d: %s" % (st, spd.spd_last_error_string(_h())))


class _Owned:
    """A library object, released with the state that holds it."""

    def __init__(self, obj, release):
        self.obj, self._release = obj, release

    def __del__(self):
        self._release(self.obj)


def prepare(case, seed):
    kind = case["kind"]
    h = _h()
    s = {"case": case}
    if kind == "batch":
        sizes, As, b, off, _ = _batch_systems(case, seed)
        x = torch.zeros_like(b)
        Bs = [b[off[i]:off[i + 1]] for i in range(len(sizes))]
        Xs = [x[off[i]:off[i + 1]] for i in range(len(sizes))]
        st, plan = spd.spd_batch_create(h, As, Bs, Xs)
        _ok(st)
        s.update(As=As, b=b, x=x, plan=_Owned(plan, spd.spd_batch_destroy))
        return s
    if kind == "learned":
        A, pts, Z, T, params = _learned_inputs(case, seed)
        st, net = spd.spd_mlp_create(h, case["hidden"], 0, case["bf16"])
        _ok(st)
        spd.spd_mlp_params(net, inp=params)
        s.update(A=A, pts=pts, Z=Z, T=T, net=_Owned(net, spd.spd_mlp_destroy), grad=torch.empty_like(params))
        return s
    A, B = _system(case, seed)
    s.update(A=A, B=B, X=torch.zeros(case["m"], case["n"], dtype=F64, device=DEV).t())
    if kind == "refine":
        st, F, _ = spd.spd_factor(h, A, case["prec"])
        _ok(st)
        s["F"] = _Owned(F, spd.spd_factor_destroy)
    return s


def run(s):
    c, h = s["case"], _h()
    kind = c["kind"]
    if kind == "solve":
        st, F, _ = spd.spd_factor(h, s["A"], c["prec"])
        _ok(st)
        st, _ = spd.spd_solve_ir(h, F, s["A"], s["B"], s["X"], {"resid": c["resid"]})
        spd.spd_factor_destroy(F)
        _ok(st)
        return s["X"]
    if kind == "refine":
        st, _ = spd.spd_solve_ir(h, s["F"].obj, s["A"], s["B"], s["X"], {"resid": c["resid"]})
        _ok(st)
        return s["X"]
    if kind == "cg":
        st, _ = spd.spd_cg(h, s["A"], s["B"], s["X"], "fp32", opts={"band": c["band"], "resid": "auto"})
        _ok(st)
        return s["X"]
    if kind == "batch":
        st, _, status, _, _ = spd.spd_batch_solve(s["plan"].obj, c["method"], c["prec"], count=c["count"])
        _ok(st)
        return s["x"], status
    F = learned.features(h, s["A"], s["pts"], c["ell"], c["nugget"])
    st, loss = spd.spd_mlp_loss_grad(s["net"].obj, s["A"], F, s["Z"], s["T"], 0.1)
    _ok(st)
    spd.spd_mlp_params(s["net"].obj, grad=s["grad"])
    return F, loss, s["grad"]


def work(case):
    """A is read once, vectors and results once; the operations of one pass of the method: a factor, two
    triangular solves and a residual (solve), the latter two (refine), one product of each kind (cg)."""
    kind = case["kind"]
    if kind == "batch":
        n = _batch_sizes(case)
        b = sum(8.0 * k * k + 16.0 * k for k in n)
        if case["method"] == "chol_ir":
            return {"bytes": b, "flops": sum(k ** 3 / 3.0 + 4.0 * k * k for k in n)}
        return {"bytes": b, "flops": sum(2.0 * k * k for k in n)}
    n = float(case["n"])
    if kind == "learned":  # two products with A; the network forward and backward
        p, H = case["p"], case["hidden"]
        net = 16 * H + H * H + 33 * H
        return {"bytes": 8.0 * n * n + 24.0 * n * p + 64.0 * n + 8.0 * net, "flops": 4.0 * n * n * p + 6.0 * n * net}
    m = case["m"]
    vec = 16.0 * n * m
    if kind == "solve":
        return {"bytes": 8.0 * n * n + vec, "flops": n ** 3 / 3.0 + 4.0 * n * n * m}
    if kind == "refine":
        return {"bytes": 10.0 * n * n + vec, "flops": 4.0 * n * n * m}
    inner = n if case["band"] < 0 else 2.0 * case["band"] + 1.0
    return {"bytes": 8.0 * n * n + 4.0 * inner * n + vec, "flops": 2.0 * (n + inner) * n * m}


# ---- the same in 64 bits, by torch alone ------------------------------------------------------------------
def _solve64(A, B):
    """A single-precision Cholesky factor of the scaled matrix and refinement in 64 bits until it no longer moves."""
    d = A.diagonal().rsqrt()
    S = torch.empty(A.shape, dtype=torch.float32, device=A.device)
    for i in range(0, A.shape[0], 4096):
        S[i:i + 4096] = (A[i:i + 4096] * d[i:i + 4096, None] * d).float()
    L = torch.linalg.cholesky(S)
    del S

    def apply(R):
        scale = R.abs().amax(0).clamp_min(1e-300)
        return d[:, None] * (torch.cholesky_solve((d[:, None] * R / scale).float(), L).double() * scale)

    X = apply(B)
    for _ in range(14):
        X = X + apply(B - A @ X)
    return X


def _rnd(x):
    return x.to(torch.bfloat16).to(F64)


def _learned64(c, seed):
    A, pts, Z, T, params = _learned_inputs(c, seed)
    n, H, p = c["n"], c["hidden"], c["p"]
    s = A.diagonal().rsqrt()
    x, y = pts[:, 0], pts[:, 1]
    Ah = (s[:, None] * A * s).abs()
    mean, rms = Ah.sum(1) / n, ((Ah ** 2).sum(1) / n).sqrt()
    Ah.fill_diagonal_(-1.0)
    mx = Ah.amax(1)
    del Ah
    one, pi = torch.ones_like(x), math.pi
    F = torch.stack([x, y, one * math.log(c["ell"]), one * math.log(c["nugget"]), torch.sin(pi * x), torch.cos(pi * x),
                     torch.sin(pi * y), torch.cos(pi * y), torch.sin(2 * pi * x), torch.cos(2 * pi * x),
                     torch.sin(2 * pi * y), torch.cos(2 * pi * y), mean, rms, mx, one], 1)
    q = _rnd if c["bf16"] else (lambda t: t)  # the bf16 network rounds the operands of its forward products
    w = params.double()
    cut = [0, 16 * H, 17 * H, 17 * H + H * H, 18 * H + H * H, 51 * H + H * H, 51 * H + H * H + 33]
    W1, b1, W2, b2, W3, b3 = (w[i:j] for i, j in zip(cut, cut[1:]))
    W1, W2, W3 = W1.view(H, 16), W2.view(H, H), W3.view(33, H)
    Fs = F.float().double()
    Z1 = q(Fs) @ q(W1).T + b1
    H1 = q(Z1 * torch.sigmoid(Z1))
    Z2 = H1 @ q(W2).T + b2
    H2 = q(Z2 * torch.sigmoid(Z2))
    O = (H2 @ q(W3).T + b3).detach().requires_grad_()
    dh, U = torch.nn.functional.softplus(O[:, 0]) + 1e-3, O[:, 1:]
    R = (s[:, None] * Z) / dh[:, None]
    C = torch.eye(32, dtype=F64, device=DEV) + U.T @ (U / dh[:, None])
    Y = s[:, None] * (R - (U / dh[:, None]) @ torch.linalg.solve(C, U.T @ R))
    E = A @ Y - Z
    loss = ((E ** 2).sum(0) / (Z ** 2).sum(0)).sum() / p + 0.1 * ((Y[:, 0] - T) ** 2).sum() / (T ** 2).sum()
    (dO,) = torch.autograd.grad(loss, O)

    def back(dH, Zk):
        t = torch.sigmoid(Zk)
        return dH * t * (1.0 + Zk * (1.0 - t))

    d2 = back(dO @ W3, Z2)
    d1 = back(d2 @ W2, Z1)
    g = [d1.T @ Fs, d1.sum(0), d2.T @ H1, d2.sum(0), dO.T @ H2, dO.sum(0)]
    return F, float(loss), torch.cat([t.reshape(-1) for t in g])


def exact(case, seed):
    if case["kind"] == "learned":
        return _learned64(case, seed)
    if case["kind"] == "batch":
        sizes, _, b, off, groups = _batch_systems(case, seed)
        x = torch.empty_like(b)
        for n, idx, A in groups:
            B = torch.stack([b[off[i]:off[i + 1]] for i in idx])[:, :, None]
            L = torch.linalg.cholesky(A)
            X = torch.cholesky_solve(B, L)
            X = X + torch.cholesky_solve(B - A @ X, L)
            for k, i in enumerate(idx):
                x[off[i]:off[i + 1]] = X[k, :, 0]
        return x, None
    A, B = _system(case, seed)
    return _solve64(A, B)
