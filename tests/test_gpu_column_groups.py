"""Many right-hand sides side by side: the super-block sweeps in groups of
columns and the digit-product residual with two column blocks per tile of A, at
the counts where the group width, the number of groups or the last group's width
changes, against the oracle's float64 results."""
import numpy as np
import pytest
import torch

import oracle
import paper_1405_4644_gb300 as spd
import workloads as W

pytestmark = pytest.mark.gpu

from tests.gpu_util import check, dev_cols, dev_sym, dev_zeros, factor_L, host  # noqa: E402
from tests.test_gpu_sb_sweeps import U32, kappa_scaled  # noqa: E402


@pytest.fixture(scope="module")
def h():
    hh = spd.spd_create(torch.cuda.current_stream())
    yield hh
    spd.spd_destroy(hh)


# one super-block, ragged; three, the last of one block of one row; a ragged fifth one
@pytest.mark.parametrize("n", [300, 2049, 4097])
def test_sweep_column_groups(h, n):
    A = W.gram_shifted(n, seed=n, shift=0.5)
    ms = (100, 2, 3, 4, 6, 9, 13, 17, 24, 25, 31, 32, 33, 48, 49, 64, 65)
    Rh = W.gaussian_rhs(n, max(ms), 11)
    st, F, _ = spd.spd_factor(h, dev_sym(A), "fp32", spd.SPD_SCALE_DIAG)
    check(h, st)
    try:
        L, d, _ = factor_L(F)
        got = {}
        for m in ms:
            Z = dev_zeros(n, m)
            check(h, spd.spd_factor_solve(h, F, dev_cols(np.asfortranarray(Rh[:, :m])), Z))
            got[m] = host(Z)
    finally:
        spd.spd_factor_destroy(F)
    ref = d[:, None] * oracle.potrs(L.T, d[:, None] * Rh)
    tol = 8.0 * U32 * n ** 0.5 * kappa_scaled(A)
    for m in ms:
        err = np.linalg.norm(got[m] - ref[:, :m], axis=0) / np.linalg.norm(ref[:, :m], axis=0)
        assert err.max() <= tol, (m, err.max(), tol)


# below one K tile and one row block; ragged in both; several row blocks a CTA
@pytest.mark.parametrize("n,ms", [(2, (17,)), (50, (17, 33)), (300, (17, 32, 33, 48, 49, 64)), (2049, (18, 40))])
def test_digit_residual_column_blocks(h, n, ms):
    """The digit sums are exact integers: a column's residual has the same bits whichever
    columns it is computed with.  16 at a time (one column block per tile of A) against
    all at once (two)."""
    At = dev_sym(W.gram_shifted(n, seed=n, shift=0.5))
    Bh, Xh = W.gaussian_rhs(n, max(ms), 5), W.gaussian_rhs(n, max(ms), 6)
    want = []
    for c in range(0, max(ms), 16):
        R = dev_zeros(n, min(16, max(ms) - c))
        check(h, spd.spd_residual_tc(h, At, dev_cols(np.asfortranarray(Bh[:, c:c + 16])),
                                     dev_cols(np.asfortranarray(Xh[:, c:c + 16])), R))
        want.append(host(R))
    want = np.concatenate(want, axis=1)
    for m in ms:
        R = dev_zeros(n, m)
        check(h, spd.spd_residual_tc(h, At, dev_cols(np.asfortranarray(Bh[:, :m])), dev_cols(np.asfortranarray(Xh[:, :m])), R))
        assert np.array_equal(host(R), want[:, :m]), m
