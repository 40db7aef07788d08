"""Batched systems with zero and non-finite right-hand sides: x = 0 for b = 0, and no
system with a NaN or an infinity in its data counts as solved."""
import numpy as np
import pytest
import torch

import paper_1405_4644_gb300 as spd
import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 31, 32, 33, 64, 200, 257, 300, 512]
METHODS = [("chol_ir", "fp32"), ("chol_ir", "bf16"), ("pcg_jacobi", "fp32")]


def solve(As, bs, method, prec, opts=None):
    h = spd.spd_create(torch.cuda.current_stream())
    dA = [torch.from_numpy(np.asfortranarray(a).T.copy()).cuda().t() for a in As]  # column-major
    db = [torch.from_numpy(b).cuda() for b in bs]
    dx = [torch.full_like(b, 7.0) for b in db]
    st, plan = spd.spd_batch_create(h, dA, db, dx)
    assert st == 0
    try:
        st, _, sts, berr, it = spd.spd_batch_solve(plan, method, prec, opts, count=len(As))
        return st, sts, berr, it, [x.cpu().numpy() for x in dx]
    finally:
        spd.spd_batch_destroy(plan)
        spd.spd_destroy(h)


@pytest.mark.parametrize("method,prec", METHODS)
def test_zero_right_hand_side(method, prec):
    As = [W.gram_shifted(n, seed=n, shift=0.5) for n in SIZES]
    bs = [np.zeros(n) if k % 2 else W.rng(k).standard_normal(n) for k, n in enumerate(SIZES)]
    st, sts, berr, it, xs = solve(As, bs, method, prec)
    assert st == spd.SPD_OK
    for k, x in enumerate(xs):
        assert sts[k] == spd.SPD_OK and berr[k] <= 1e-14
        if k % 2:
            assert berr[k] == 0.0 and np.array_equal(x, np.zeros_like(x)), k
        else:
            assert np.all(np.isfinite(x)) and np.any(x)


@pytest.mark.parametrize("method,prec", METHODS)
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("where", ["b", "A"])
def test_non_finite_data_are_not_solved(method, prec, value, where):
    As = [W.gram_shifted(n, seed=n, shift=0.5) for n in SIZES]
    bs = [W.rng(k).standard_normal(n) for k, n in enumerate(SIZES)]
    hit = [k for k, n in enumerate(SIZES) if k % 2 and n > 1]
    for k in hit:
        n = SIZES[k]
        if where == "b":
            bs[k][n // 2] = value
        else:  # above the diagonal: the factor does not read it, the residual does
            As[k][0, n - 1] = value
    st, sts, berr, it, xs = solve(As, bs, method, prec, {"maxit_inner": 300})
    assert st == spd.SPD_ERR_NO_CONVERGENCE
    for k in range(len(SIZES)):
        if k in hit:
            assert sts[k] == spd.SPD_ERR_NO_CONVERGENCE and not berr[k] <= 1e-14, k
        else:
            assert sts[k] == spd.SPD_OK and berr[k] <= 1e-14 and np.all(np.isfinite(xs[k])), k
