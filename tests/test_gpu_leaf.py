"""The 128 x 128 leaf of the float32 factor: where its micro-steps, steps and
barriers meet, the pivots that break down, and subnormal pivots."""
import numpy as np
import pytest

import oracle
import paper_1405_4644_gb300 as spd
import workloads as W

pytestmark = pytest.mark.gpu

from tests.gpu_util import check, dev_sym, factor_L  # noqa: E402


@pytest.fixture(scope="module")
def h():
    import torch
    hh = spd.spd_create(torch.cuda.current_stream())
    yield hh
    spd.spd_destroy(hh)


@pytest.mark.parametrize("n", [4, 5, 32, 36, 63, 64, 65, 96, 100, 125, 126, 160, 255, 256])
def test_leaf_edges(h, n):
    A = W.gram_shifted(n, seed=n, shift=0.3)
    d = 1.0 / np.sqrt(np.diag(A))
    As = d[:, None] * A * d
    st, F, _ = spd.spd_factor(h, dev_sym(A), "fp32")
    check(h, st)
    L, _, _ = factor_L(F)
    spd.spd_factor_destroy(F)
    # a float32 factor: ||L L^T - As|| <= c n 2^-24 ||As||, forward kappa times that
    u, k = 2.0 ** -24, np.linalg.cond(As)
    assert np.linalg.norm(L @ L.T - As) <= 4 * max(n, 8) ** 0.5 * u * np.linalg.norm(As)
    R = oracle.potrf(As).T
    assert np.max(np.abs(L - R)) <= 8 * k * max(n, 8) ** 0.5 * u * np.max(np.abs(R))


@pytest.mark.parametrize("col", [1, 3, 4, 5, 31, 32, 35, 63, 64, 95, 96, 126, 127, 130])
def test_breakdown_names_the_column(h, col):
    A = np.eye(140)
    A[col, col - 1] = A[col - 1, col] = 1.5  # pivot of `col`: 1 - 2.25
    st, F, rep = spd.spd_factor(h, dev_sym(A), "fp32")
    assert st == spd.SPD_ERR_NOT_SPD and F is None
    assert rep.info == col + 1


@pytest.mark.parametrize("col", [0, 2, 33, 127])
def test_subnormal_pivot(h, col):
    """Without the diagonal scaling a pivot may be subnormal in float32: its square root is still taken."""
    n = 130
    A = np.eye(n)
    A[col, col] = 2.0 ** -140
    st, F, _ = spd.spd_factor(h, dev_sym(A), "fp32", flags=0)
    check(h, st)
    L, _, _ = factor_L(F)
    spd.spd_factor_destroy(F)
    want = np.eye(n)
    want[col, col] = 2.0 ** -70
    assert np.max(np.abs(L - want) / np.where(want > 0, want, 1.0)) <= 2.0 ** -21


@pytest.mark.parametrize("n", [129, 200, 256, 257, 383, 385, 512, 640, 769, 897, 1023, 1024])
@pytest.mark.parametrize("m", [1, 2, 17])
def test_one_super_block(h, n, m):
    """Orders of one super-block: the sweep is the product with its inverse, formed by doubling."""
    import torch
    A = W.gram_shifted(n, seed=n, shift=0.1)
    At = dev_sym(A)
    st, F, _ = spd.spd_factor(h, At, "fp32")
    check(h, st)
    L, d, _ = factor_L(F)
    R = torch.from_numpy(W.gaussian_rhs(n, m, 3).T.copy()).to(At.device).t()
    Z = torch.zeros_like(R)
    check(h, spd.spd_factor_solve(h, F, R, Z))
    spd.spd_factor_destroy(F)
    Lt = np.linalg.inv(L)
    want = d[:, None] * (Lt.T @ (Lt @ (d[:, None] * R.cpu().numpy())))
    # float32 products with an explicit float32 inverse: n^1/2 2^-24 times cond(L) squared
    tol = 8 * n ** 0.5 * 2.0 ** -24 * np.linalg.cond(L) ** 2
    assert np.linalg.norm(Z.cpu().numpy() - want) <= tol * np.linalg.norm(want)


@pytest.mark.parametrize("e", [-140, -127, -126, -125, 0, 123, 124, 125, 126])
def test_conversion_at_the_ends_of_the_exponent_range(h, e):
    """A diagonal matrix without scaling: its entries reach the leaf by the conversion alone."""
    n = 70
    m = np.where(np.arange(n) % 3 == 0, 1.0, np.where(np.arange(n) % 3 == 1, 1.5, 1.9375))  # short: exact as subnormals
    a = m * 2.0 ** e
    st, F, _ = spd.spd_factor(h, dev_sym(np.diag(a)), "fp32", flags=0)
    check(h, st)
    L, _, _ = factor_L(F)
    spd.spd_factor_destroy(F)
    # three roundings of 2^-24 in the conversion (none here), one square root and one product
    assert np.max(np.abs(np.diag(L) / np.sqrt(a) - 1.0)) <= 2.0 ** -21


@pytest.mark.parametrize("n", [200, 1024])
def test_one_super_block_under_a_memory_cap(h, n):
    """A cap that holds the factor but not its super-block's inverse: the block sweeps serve."""
    import torch
    A = W.gram_shifted(n, seed=n, shift=0.5)
    At = dev_sym(A)
    B = torch.from_numpy(W.gaussian_rhs(n, 1, 3).T.copy()).to(At.device).t()
    nb, ldw = -(-n // 128), -(-n // 64) * 64
    need = 8 * n + 4 * (n * ldw + 86016 * nb) + 6 * n * ldw  # d, W, the blocks' inverses and couplings, the mirror
    X = {}
    try:
        for cap in (0, need):
            spd.spd_set_memory_cap(h, cap)
            st, F, _ = spd.spd_factor(h, At, "fp32")
            check(h, st)
            spd.spd_set_memory_cap(h, 0)
            Z = torch.zeros_like(B)
            check(h, spd.spd_factor_solve(h, F, B, Z))
            spd.spd_factor_destroy(F)
            X[cap] = Z.cpu().numpy()
    finally:
        spd.spd_set_memory_cap(h, 0)
    ref = np.linalg.solve(A, B.cpu().numpy())
    tol = 8 * n ** 0.5 * 2.0 ** -24 * np.linalg.cond(A)  # as two float32 solves
    for x in X.values():
        assert np.linalg.norm(x - ref) <= tol * np.linalg.norm(ref)
