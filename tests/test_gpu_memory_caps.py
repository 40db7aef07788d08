"""Calls under a memory cap that leaves room for what they cannot do without: partial
sums that only serve speed are left out, and the call is served."""
import numpy as np
import pytest
import torch

import paper_1405_4644_gb300 as spd
import workloads as W
from tests.gpu_util import dev_cols, dev_sym, dev_zeros
from tests.test_gpu_learned_shapes import loss64

pytestmark = pytest.mark.gpu


def total(*sizes):
    """Bytes of a workspace of these arrays, each on a 256-byte boundary."""
    return sum((s + 255) // 256 * 256 for s in sizes)


@pytest.mark.parametrize("n,p,H", [(1, 1, 8), (33, 3, 16), (700, 17, 130), (1023, 8, 64)])
def test_training_step(n, p, H):
    # vectors of the loss, projections, the preconditioner
    request = total(8 * n, *[8 * n * p] * 7, 8 * 32 * p, 8 * 32 * p, 8 * -(-n // 256) * 32 * p, 8 * (2 * p + 2), 8 * p,
                    8 * n, 8 * 32 * n, 8 * 2048, 4)
    A = W.matern32_torch(W.matern_points(n, 5), 0.2, 0.1, "cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(n + p)
    F = torch.rand(n, 16, device="cuda", generator=g)
    Z = torch.randn(p, n, dtype=torch.float64, device="cuda", generator=g).t()
    T = torch.linalg.solve(A, Z[:, 0]).contiguous()
    h = spd.spd_create(torch.cuda.current_stream())
    try:
        st, net = spd.spd_mlp_create(h, H, 3, False)
        assert st == spd.SPD_OK
        cnt = spd.spd_mlp_params(net)
        params = 0.2 * torch.randn(cnt, device="cuda", generator=g)
        spd.spd_mlp_params(net, inp=params)
        L64, g64 = loss64(torch, params, H, A, F, Z, T, 0.1)
        tol = 2.0 ** -21 * 6 * 100  # as in test_gpu_learned_shapes.test_gradient
        for cap, want in [(request - 1, spd.SPD_ERR_OOM), (request, spd.SPD_OK), (0, spd.SPD_OK)]:
            spd.spd_set_memory_cap(h, cap)
            st, L = spd.spd_mlp_loss_grad(net, A, F, Z, T, 0.1)
            assert st == want, cap
            if st == spd.SPD_OK:
                grad = torch.empty(cnt, device="cuda")
                spd.spd_mlp_params(net, grad=grad)
                assert abs(L - L64) <= tol * abs(L64)
                assert float((grad.double() - g64).norm()) <= tol * float(g64.norm())
        spd.spd_mlp_destroy(net)
    finally:
        spd.spd_destroy(h)


def solver_request(n, m):
    """spd_solve_ir with the float64 residual: the residual's partial sums, eight vectors of
    n m and float32 copies, one pair of dot partials per row chunk and column, the
    columns' state."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = -(-n // 256)
    split = min(max(1, (4 * sms + blocks - 1) // blocks), max(1, n // 256))  # float64 kernel
    best, best_eff = 1, -1.0  # float32-pair kernel
    for s in range(1, max(1, n // 128) + 1):
        ctas = blocks * s
        eff = ctas / (-(-ctas // (2 * sms)) * 2 * sms)
        if ctas < 4 * sms and s < max(1, n // 128):
            eff *= 0.5
        if eff > best_eff + 1e-9:
            best, best_eff = s, eff
        if ctas >= 8 * sms:
            break
    split = max(split, best)
    dots = max(1, min(2 * sms, blocks) // m)
    nm = n * m
    return [8 * split * nm, 4 * split * n, 8 * 3 * blocks * m, 16 * m, 8 * nm, 24 * m, 8, 8 * m, 8 * m, *[8 * nm] * 5,
            16 * dots * m, 8 * nm, 4 * nm, 32 * m, 32, 56 * m, 4 * m, 4]


SHAPES = [(1, 1), (2, 40), (2, 3), (3, 9), (4, 8), (33, 8), (300, 1), (2000, 8), (2000, 33), (3000, 16)]


@pytest.mark.parametrize("n,m", SHAPES)
def test_refinement(n, m):
    A = W.gram_shifted(n, seed=n, shift=0.5)
    Ad, Bd, X = dev_sym(A), dev_cols(W.gaussian_rhs(n, m, 1)), dev_zeros(n, m)
    h = spd.spd_create(torch.cuda.current_stream())
    try:
        st, F, _ = spd.spd_factor(h, Ad, "fp32")
        assert st == spd.SPD_OK
        spd.spd_set_memory_cap(h, total(*solver_request(n, m)))
        st, rep = spd.spd_solve_ir(h, F, Ad, Bd, X, {"resid": "fp64"})
        assert st == spd.SPD_OK and rep.berr <= 1e-14
        spd.spd_factor_destroy(F)
    finally:
        spd.spd_destroy(h)


@pytest.mark.parametrize("kind", ["fp32", "bf16", "fp64", "band", "jacobi"])
@pytest.mark.parametrize("n,m", SHAPES)
def test_cg(n, m, kind):
    # the inner matrix: float32 (rows to a multiple of 64), bf16, a band of half-width 3 or none
    inner = {"fp32": 4 * n * (-(-n // 64) * 64), "bf16": 2 * n * (-(-n // 64) * 64), "fp64": 0, "band": 4 * 7 * n,
             "jacobi": 4 * 7 * n}[kind]
    A = W.gram_shifted(n, seed=n, shift=2.0)
    if kind in ("band", "jacobi"):
        i = np.arange(n)
        A = np.where(np.abs(i[:, None] - i) <= 3, A, 0.0)
        A[i, i] = 8.0 + i / n
    Ad, Bd, X = dev_sym(A), dev_cols(W.gaussian_rhs(n, m, 1)), dev_zeros(n, m)
    extra = [8 * n] if kind == "jacobi" else []
    opts = {"resid": "fp64", "matvec_cores": "cuda" if kind == "fp32" else "auto"}
    if kind in ("band", "jacobi"):
        opts["band"] = 3
    h = spd.spd_create(torch.cuda.current_stream())
    try:
        spd.spd_set_memory_cap(h, total(*solver_request(n, m), inner, *extra))
        st, rep = spd.spd_cg(h, Ad, Bd, X, kind if kind in ("fp32", "bf16", "fp64") else "fp32",
                             pc="jacobi" if kind == "jacobi" else "none", opts=opts)
        assert st == spd.SPD_OK and rep.berr <= 1e-14
        R = np.abs(Bd.cpu().numpy() - A @ X.cpu().numpy()).max(0)
        assert np.all(R <= (1e-14 + n * 2.0**-53) * np.abs(A).sum(1).max() * np.abs(X.cpu().numpy()).max(0))
    finally:
        spd.spd_destroy(h)


def test_batched_plan():
    """One CTA's scratch per SM, and as many CTAs, where two per SM are over the cap; a plan
    is never refused for it."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sizes = [16 + (7 * k) % 100 for k in range(4 * sms)]
    dA = [torch.from_numpy(W.gram_shifted(n, seed=k, shift=0.5)).cuda() for k, n in enumerate(sizes)]
    db = [torch.from_numpy(W.rng(k).standard_normal(n)).cuda() for k, n in enumerate(sizes)]
    want = None
    for cap, most in [(0, 2 * sms), (sms << 20, sms), (1 << 16, sms)]:
        h = spd.spd_create(torch.cuda.current_stream())
        try:
            spd.spd_set_memory_cap(h, cap)
            dx = [torch.zeros_like(b) for b in db]
            free = torch.cuda.mem_get_info()[0]
            st, plan = spd.spd_batch_create(h, dA, db, dx)
            assert st == spd.SPD_OK
            used = free - torch.cuda.mem_get_info()[0]
            assert used <= (most << 20) + (32 << 20)  # the tables, and the driver's granularity
            for method in ("chol_ir", "pcg_jacobi"):
                st, _, sts, berr, _ = spd.spd_batch_solve(plan, method, "fp32", count=len(sizes))
                assert st == spd.SPD_OK and np.all(berr[:len(sizes)] <= 1e-14)
                if method == "chol_ir":
                    assert spd.spd_batch_info(plan, method)["ctas"] <= most
                    xs = [x.cpu().numpy() for x in dx]
                    want = want or xs
                    assert all(np.array_equal(a, b) for a, b in zip(xs, want))
            spd.spd_batch_destroy(plan)
        finally:
            spd.spd_destroy(h)
