"""CG steps whose launches are fused: the banded product with the p-update (both
sides of its band limit, ragged ends, several columns, with and without Jacobi),
the products that write their own share of p^T q, and the norm of A."""
import numpy as np
import pytest

import oracle
import paper_1405_4644_gb300 as spd
import workloads as W

pytestmark = pytest.mark.gpu

from tests.gpu_util import check, dev_cols, dev_sym, dev_zeros, host  # noqa: E402


@pytest.fixture(scope="module")
def h():
    import torch
    hh = spd.spd_create(torch.cuda.current_stream())
    yield hh
    spd.spd_destroy(hh)


def solve(h, A, B, mv, **kw):
    X = dev_zeros(*B.shape)
    st, rep = spd.spd_cg(h, dev_sym(A), dev_cols(B), X, mv, **kw)
    check(h, st)
    return host(X), rep


def bound(A, B, X):
    """berr <= 1e-14 is the rule; the solution then errs by at most kappa 1e-14 of the norm ratio."""
    want = oracle.solve(A, B)
    err = np.max(np.abs(X - want)) / np.max(np.abs(want))
    assert err <= 2 * np.linalg.cond(A, np.inf) * 1e-14, err


@pytest.mark.parametrize("pc", ["none", "jacobi"])
@pytest.mark.parametrize("n,m,band", [(1, 1, 0), (5, 2, 3), (127, 1, 16), (128, 3, 0), (129, 1, 128), (700, 9, 5),
                                      (700, 33, 255), (700, 1, 256), (700, 2, 257), (1000, 1, 33)])
def test_banded_step(h, n, m, band, pc):
    A = W.model_covariance(n, 4)
    B = W.uniform_rhs(n, m, 3)
    X, rep = solve(h, A, B, "fp32", pc=pc, opts={"band": band, "maxit": 200})
    bound(A, B, X)
    assert rep.iters_low >= 1


@pytest.mark.parametrize("mv,m", [("fp32", 1), ("fp32", 4), ("fp32", 7), ("bf16", 5), ("bf16", 8), ("bf16", 9),
                                  ("fp32", 8), ("fp32", 31), ("fp32", 33), ("fp32", 65)])
@pytest.mark.parametrize("n", [31, 33, 513])
def test_products_with_their_dots(h, n, m, mv):
    A = W.model_covariance(n, 2)
    B = W.uniform_rhs(n, m, 7)
    X, _ = solve(h, A, B, mv, pc="jacobi", opts={"maxit": 200})
    bound(A, B, X)


@pytest.mark.parametrize("n", [1, 255, 256, 257, 1100])
def test_backward_error_uses_the_norm_of_a(h, n):
    """The reported backward error, recomputed from the solution: the norm of A in it is right to float32."""
    A = W.model_covariance(n, 1)
    B = W.uniform_rhs(n, 1, 1)
    for resid in ("fp64", "tc"):
        X = dev_zeros(n, 1)
        st, rep = spd.spd_cg(h, dev_sym(A), dev_cols(B), X, "fp32",
                             opts={"tol": 1e-3, "eta": 0.5, "maxit": 200, "resid": resid})
        check(h, st)
        x = host(X)
        want = np.max(np.abs(B - A @ x)) / (np.max(np.sum(np.abs(A), axis=1)) * np.max(np.abs(x)))
        # float32 sums of up to n terms in the norm, float64 rounding of the residual
        assert abs(rep.berr - want) <= (n * 2.0 ** -24) * want + 1e-15
