"""Batched Cholesky-IR where nearly every system breaks down, at every block of the
factor: each CTA goes from a breakdown straight to its next system many times."""
import re
from pathlib import Path

import numpy as np
import pytest
import torch

import paper_1405_4644_gb300 as spd
import workloads as W

KERNEL = Path(__file__).resolve().parent.parent / "paper_1405_4644_gb300" / "csrc" / "k_batched.cuh"


def test_the_breakdown_flag_is_read_behind_a_barrier():
    """The flag that warp 0 raises is not read between the end of one block and the
    barrier after the next diagonal block (a warp that saw it early left the loop while
    the others waited at that barrier)."""
    src = re.sub(r"//[^\n]*", "", KERNEL.read_text())
    body = src[src.index("k_batch_chol_ir(BatchArgs a)"):]
    loop = re.search(r"for \(int kb = 0;[^)]*\) \{", body)
    assert "s_bad" not in loop.group(0)
    reads = [m.start() for m in re.finditer(r"if \(s_bad\)", body)]
    assert len(reads) == 2
    between = body[loop.end():reads[0]]
    assert "__syncthreads();" in between[between.rindex("s_bad = 1"):]


@pytest.mark.gpu
def test_systems_after_breakdowns():
    h = spd.spd_create(torch.cuda.current_stream())
    As, bs, bad = [], [], []
    for k in range(1200):
        n = 33 + (k * 37) % 400
        A = np.eye(n)
        if k % 8:  # pivot q is 1 - 2.25, q from the first block to the last
            q = 1 + (k * 53) % (n - 1)
            A[q, q - 1] = A[q - 1, q] = 1.5
        else:
            A = W.gram_shifted(n, seed=k, shift=0.5)
        bad.append(bool(k % 8))
        As.append(A)
        bs.append(W.rng(k).standard_normal(n))
    dA = [torch.from_numpy(a).cuda() for a in As]
    db = [torch.from_numpy(b).cuda() for b in bs]
    dx = [torch.zeros_like(b) for b in db]
    st, plan = spd.spd_batch_create(h, dA, db, dx)
    assert st == 0
    try:
        for _ in range(3):
            st, rep, sts, berr, it = spd.spd_batch_solve(plan, "chol_ir", "fp32", count=len(As))
            assert st == spd.SPD_ERR_NOT_SPD
            for k in range(len(As)):
                assert sts[k] == (spd.SPD_ERR_NOT_SPD if bad[k] else spd.SPD_OK), k
                if not bad[k]:
                    assert berr[k] <= 1e-14
                    x, want = dx[k].cpu().numpy(), np.linalg.solve(As[k], bs[k])
                    tol = 2 * np.linalg.cond(As[k], np.inf) * 1e-14  # berr <= 1e-14, and LAPACK's own error
                    assert np.max(np.abs(x - want)) <= tol * np.max(np.abs(want)), k
    finally:
        spd.spd_batch_destroy(plan)
        spd.spd_destroy(h)
