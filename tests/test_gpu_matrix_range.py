"""||A||_inf over the whole range of float64: refinement of matrices whose entries are
below, above or across the range of float32 stops at the backward error it reports."""
import numpy as np
import pytest

import paper_1405_4644_gb300 as spd
import workloads as W
from tests.gpu_util import dev_cols, dev_sym, dev_zeros, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    hh = spd.spd_create()
    yield hh
    spd.spd_destroy(hh)


def solve(h, A, B, resid, prec="bf16"):
    n, m = B.shape
    Ad, X = dev_sym(A), dev_zeros(n, m)
    st, F, _ = spd.spd_factor(h, Ad, prec)
    assert st == spd.SPD_OK
    try:
        st, rep = spd.spd_solve_ir(h, F, Ad, dev_cols(B), X, {"resid": resid})
    finally:
        spd.spd_factor_destroy(F)
    return st, rep, host(X)


def backward_error(A, B, X, k):
    """max_c ||b - A x||_inf / (||A||_inf ||x||_inf) in extended precision, for A, B scaled back by 2^-k."""
    A, B = np.ldexp(A, -k).astype(np.longdouble), np.ldexp(B, -k).astype(np.longdouble)
    R = np.abs(B - A @ X.astype(np.longdouble)).max(0)
    return float((R / (np.abs(A).sum(1).max() * np.abs(X).max(0))).max())


# float32: normal from 2^-126, subnormal from 2^-149, up to 2^128.  The corrections are
# solved for in float32 from D r, of the size 2^(k / 2) |b|, which has to keep 53 bits
# below it in float32's normal range: |k| <= 146
@pytest.mark.parametrize("k", [-146, -140, -130, -120, 0, 120, 130, 146])
@pytest.mark.parametrize("resid,n,m", [("fp64", 333, 1), ("fp64", 700, 3), ("tc", 700, 3), ("tc", 333, 18),
                                       ("df32", 700, 3)])
def test_scaled_by_a_power_of_two(h, resid, n, m, k):
    A = W.gram_shifted(n, seed=n, shift=0.2)
    B = A @ W.gaussian_rhs(n, m, 3)  # on the scale of A, so that an absolute test would accept at once
    A, B = np.ldexp(A, k), np.ldexp(B, k)
    st, rep, X = solve(h, A, B, resid)
    assert st == spd.SPD_OK
    be = backward_error(A, B, X, k)
    assert be <= 1e-14
    # the reported value: its norm is a sum of |a| rounded (or truncated) to 24 bits and
    # summed in float32, and its residual is rounded to float64 (relative to |A||x|: n 2^-53)
    assert abs(rep.berr - be) <= 1e-3 * be + n * 2.0**-53
    assert rep.berr > 0.0


@pytest.mark.parametrize("resid", ["fp64", "tc"])
def test_rows_across_the_range_of_float32(h, resid):
    """One row above float32's range beside ordinary ones, and one below among them."""
    n = 300
    A = W.gram_shifted(n, seed=7, shift=0.5)
    s = np.ones(n)
    s[5], s[200] = 2.0**68, 2.0**-70  # diagonal entries near 2^136 and 2^-140
    A = s[:, None] * A * s
    B = A @ W.gaussian_rhs(n, 2, 4)
    st, rep, X = solve(h, A, B, resid)
    assert st == spd.SPD_OK
    be = backward_error(A, B, X, 0)
    assert 0.0 < rep.berr <= 1e-14 and abs(rep.berr - be) <= 1e-3 * be + n * 2.0**-53
