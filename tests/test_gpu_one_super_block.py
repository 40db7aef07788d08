"""Factors of one super-block (2 to 8 blocks): their sweeps are ordinary kernels, which run
beside another stream's work, and a captured solve replays."""
import numpy as np
import pytest
import torch

import oracle
import paper_1405_4644_gb300 as spd
import workloads as W
from tests.gpu_util import check, dev_cols, dev_sym, dev_zeros, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(1000, 64), (300, 20)])
def test_sweeps_do_not_wait_for_the_whole_gpu(n, m):
    """One warp of another stream keeps an SM from a sweep's CTA (whose registers fill an
    SM) for half a second; the sweeps are over long before it ends."""
    other, s = torch.cuda.Stream(), torch.cuda.Stream()
    h = spd.spd_create(s)
    try:
        A = W.gram_shifted(n, seed=3, shift=0.1)
        with torch.cuda.stream(s):
            Ad, R, Z = dev_sym(A), dev_cols(W.gaussian_rhs(n, m, 1)), dev_zeros(n, m)
            Z0 = dev_zeros(n, m)
            st, F, _ = spd.spd_factor(h, Ad, "fp32")
            check(h, st)
            check(h, spd.spd_factor_solve(h, F, R, Z0))  # sizes the scratch
        torch.cuda.synchronize()
        done = torch.cuda.Event()
        with torch.cuda.stream(other):
            torch.cuda._sleep(1_000_000_000)
            done.record()
        check(h, spd.spd_factor_solve(h, F, R, Z))  # returns when it is done
        assert not done.query()
        torch.cuda.synchronize()
        assert torch.equal(Z, Z0)
        spd.spd_factor_destroy(F)
    finally:
        spd.spd_destroy(h)


@pytest.mark.parametrize("n,m,resid", [(129, 1, "fp64"), (1000, 1, "fp64"), (1000, 5, "tc"), (1024, 40, "tc")])
def test_captured_solve_replays(n, m, resid):
    s = torch.cuda.Stream()
    h = spd.spd_create(s)
    try:
        A = W.gram_shifted(n, seed=22, shift=0.1)
        buf = spd.spd_report_dev_buffer()
        opts = {"resid": resid, "maxit": 12}
        with torch.cuda.stream(s):
            Ad, Bd, X = dev_sym(A), dev_zeros(n, m), dev_zeros(n, m)
            st, F, _ = spd.spd_factor(h, Ad, "fp16")
            check(h, st)
            check(h, spd.spd_solve_ir_async(h, F, Ad, Bd, X, buf, opts))  # sizes the workspace
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            st = spd.spd_solve_ir_async(h, F, Ad, Bd, X, buf, opts)
        check(h, st)
        for seed in (2, 3):
            Bh = W.gaussian_rhs(n, m, seed)
            with torch.cuda.stream(s):
                Bd.copy_(dev_cols(Bh))
                X.zero_()
                g.replay()
            s.synchronize()
            r = spd.spd_report_dev_read(buf)
            assert r.status == spd.SPD_OK and r.active == 0 and r.dev_flags == 0
            assert oracle.berr(A, Bh, host(X)) <= 1e-14
        spd.spd_factor_destroy(F)
    finally:
        spd.spd_destroy(h)
