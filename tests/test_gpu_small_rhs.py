"""Right-hand sides far below 1: the backward error is relative, so x = 0 is no answer
to them."""
import numpy as np
import pytest
import torch

import paper_1405_4644_gb300 as spd
import workloads as W
from tests.gpu_util import dev_cols, dev_sym, dev_zeros, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    hh = spd.spd_create()
    yield hh
    spd.spd_destroy(hh)


@pytest.mark.parametrize("m,band", [(1, -1), (3, -1), (9, -1), (2, 8)])
def test_cg(h, m, band):
    n = 300
    i = np.arange(n)
    A = 1.0 / np.maximum(np.abs(i[:, None] - i), 1) ** 4.0
    np.fill_diagonal(A, 1.0 + np.sqrt(i + 1.0))
    B = W.rng(3).random((n, m))
    B[:, 0] *= 1e-16  # ||b - A 0|| is below the tolerance of 1e-14 in absolute terms
    X = dev_zeros(n, m)
    st, rep = spd.spd_cg(h, dev_sym(A), dev_cols(B), X, "fp32", opts={"band": band})
    assert st == spd.SPD_OK
    X = host(X)
    R = np.abs(B - A @ X).max(0) / (np.abs(A).sum(1).max() * np.abs(X).max(0))
    # berr <= 1e-14 and the check's own rounding of A X
    assert np.all(R <= 1e-14 + n * 2.0**-53)


@pytest.mark.parametrize("method", ["chol_ir", "pcg_jacobi"])
def test_batched(h, method):
    sizes = [1, 5, 64, 300]
    As = [W.gram_shifted(n, seed=n, shift=0.5) for n in sizes]
    bs = [1e-16 * W.rng(n).standard_normal(n) for n in sizes]
    dA = [torch.from_numpy(a).cuda() for a in As]
    db = [torch.from_numpy(b).cuda() for b in bs]
    dx = [torch.zeros_like(b) for b in db]
    st, plan = spd.spd_batch_create(h, dA, db, dx)
    assert st == 0
    try:
        st, _, sts, berr, _ = spd.spd_batch_solve(plan, method, "fp32", count=len(sizes))
        assert st == spd.SPD_OK
        for A, b, x in zip(As, bs, dx):
            x = x.cpu().numpy()
            r = np.abs(b - A @ x).max() / (np.abs(A).sum(1).max() * np.abs(x).max())
            assert r <= 1e-14 + len(b) * 2.0**-53
    finally:
        spd.spd_batch_destroy(plan)
