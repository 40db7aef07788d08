"""Batched systems at the edges of the kernels' tiles (32-row blocks, 256 and 512
threads a row each), with systems that break down among them."""
import numpy as np
import pytest
import torch

import paper_1405_4644_gb300 as spd
import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 4, 5, 31, 32, 33, 35, 36, 63, 64, 65, 96, 127, 128, 129, 255, 256, 257, 288, 300, 480, 481, 511, 512]


@pytest.fixture(scope="module")
def h():
    hh = spd.spd_create(torch.cuda.current_stream())
    yield hh
    spd.spd_destroy(hh)


@pytest.mark.parametrize("method,prec", [("chol_ir", "fp32"), ("chol_ir", "bf16"), ("chol_ir", "fp16"),
                                         ("pcg_jacobi", "fp32")])
def test_sizes_and_breakdowns(h, method, prec):
    As, bs, bad = [], [], {}
    for k, n in enumerate(SIZES):
        A = W.gram_shifted(n, seed=k, shift=0.5)
        if method == "chol_ir" and n in (36, 65, 300, 512):  # pivot n - 1 is 1 - 2.25
            A = np.eye(n)
            A[n - 1, n - 2] = A[n - 2, n - 1] = 1.5
            bad[k] = n
        As.append(A)
        bs.append(W.rng(100 + k).standard_normal(n))
    dA = [torch.from_numpy(a).cuda() for a in As]
    db = [torch.from_numpy(b).cuda() for b in bs]
    dx = [torch.zeros_like(b) for b in db]
    st, plan = spd.spd_batch_create(h, dA, db, dx)
    assert st == 0
    try:
        for _ in range(2):  # the second replays the tuned graph over used scratch
            st, rep, sts, berr, it = spd.spd_batch_solve(plan, method, prec, count=len(As))
            assert st == (spd.SPD_ERR_NOT_SPD if bad else spd.SPD_OK)
            for k, (A, b) in enumerate(zip(As, bs)):
                if k in bad:
                    assert sts[k] == spd.SPD_ERR_NOT_SPD
                    continue
                assert sts[k] == 0 and berr[k] <= 1e-14
                x, want = dx[k].cpu().numpy(), np.linalg.solve(A, b)
                # berr <= 1e-14: the solution within kappa_inf 1e-14, and LAPACK's own error
                tol = 2 * np.linalg.cond(A, np.inf) * 1e-14
                assert np.max(np.abs(x - want)) <= tol * np.max(np.abs(want)), (k, len(b))
    finally:
        spd.spd_batch_destroy(plan)
