"""A NaN or an infinity in the right-hand sides or in the part of A that only the
residual reads: the columns it reaches are not solved, the others are."""
import numpy as np
import pytest
import torch

import paper_1405_4644_gb300 as spd
import workloads as W
from tests.gpu_util import dev_cols, dev_sym, dev_zeros, host

pytestmark = pytest.mark.gpu

N, M = 300, 3
RESID = ["fp64", "tc", "df32"]


@pytest.fixture(scope="module")
def h():
    hh = spd.spd_create()
    yield hh
    spd.spd_destroy(hh)


def data(value, where):
    A = W.gram_shifted(N, seed=1, shift=0.3)
    B = W.gaussian_rhs(N, M, 2)
    Aw = A.copy()
    if where == "b":
        B[17, 1] = value
    else:
        Aw[N - 1, 0] = value  # row-major: above the diagonal of the column-major reading
    return A, Aw, B


def backward_errors(A, B, X):
    R = np.abs(B - A @ X).max(0)
    return R / (np.abs(A).sum(1).max() * np.abs(X).max(0))


@pytest.mark.parametrize("resid", RESID)
@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("where", ["b", "A"])
def test_refinement(h, where, value, resid):
    A, Aw, B = data(value, where)
    Ad, X = dev_sym(Aw), dev_zeros(N, M)
    st, F, _ = spd.spd_factor(h, Ad, "bf16")
    assert st == spd.SPD_OK
    try:
        st, rep = spd.spd_solve_ir(h, F, Ad, dev_cols(B), X, {"resid": resid})
    finally:
        spd.spd_factor_destroy(F)
    assert st == spd.SPD_ERR_NO_CONVERGENCE and rep.berr == np.inf
    if where == "b":
        be = backward_errors(A, B[:, [0, 2]], host(X)[:, [0, 2]])
        assert be.max() <= 1e-14


@pytest.mark.parametrize("crit", [0, 1, 2])
def test_every_criterion(h, crit):
    A, Aw, B = data(np.nan, "b")
    Ad, X = dev_sym(Aw), dev_zeros(N, M)
    st, F, _ = spd.spd_factor(h, Ad, "fp32")
    assert st == spd.SPD_OK
    try:
        st, rep = spd.spd_solve_ir(h, F, Ad, dev_cols(B), X, {"crit": crit, "tol": 1e-10})
    finally:
        spd.spd_factor_destroy(F)
    assert st == spd.SPD_ERR_NO_CONVERGENCE
    assert backward_errors(A, B[:, [0, 2]], host(X)[:, [0, 2]]).max() <= 1e-10


@pytest.mark.parametrize("resid", ["fp64", "tc"])
def test_capturable_solve(resid):
    s = torch.cuda.Stream()
    h = spd.spd_create(s)
    try:
        A, Aw, B = data(np.nan, "b")
        buf = spd.spd_report_dev_buffer()
        with torch.cuda.stream(s):
            Ad, Bd, X = dev_sym(Aw), dev_cols(B), dev_zeros(N, M)
            st, F, _ = spd.spd_factor(h, Ad, "fp32")
            assert st == spd.SPD_OK
            assert spd.spd_solve_ir_async(h, F, Ad, Bd, X, buf, {"resid": resid, "maxit": 8}) == spd.SPD_OK
        s.synchronize()
        r = spd.spd_report_dev_read(buf)
        assert r.status == spd.SPD_ERR_NO_CONVERGENCE and r.active == 1
        spd.spd_factor_destroy(F)
    finally:
        spd.spd_destroy(h)


@pytest.mark.parametrize("band", [-1, 4])
def test_cg(h, band):
    A, Aw, B = data(np.nan, "b")
    X = dev_zeros(N, M)
    st, rep = spd.spd_cg(h, dev_sym(Aw), dev_cols(B), X, "fp32", opts={"band": band, "maxit": 30})
    assert st == spd.SPD_ERR_NO_CONVERGENCE
    if band < 0:
        assert backward_errors(A, B[:, [0, 2]], host(X)[:, [0, 2]]).max() <= 1e-14
