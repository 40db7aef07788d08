"""The learned preconditioner's row features are those of the scaled matrix: a power of
four on the whole matrix changes no bit of them, to the ends of float64's range."""
import numpy as np
import pytest
import torch

import paper_1405_4644_gb300 as spd
import workloads as W
from tests.gpu_util import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 33, 300])
def test_scaled_matrices(n):
    h = spd.spd_create(torch.cuda.current_stream())
    try:
        pts = W.matern_points(n, 2)
        A = W.matern32_torch(pts, 0.1, 0.05, "cuda")
        P = torch.from_numpy(pts).to("cuda")
        out = {}
        for k in (0, -1000, -500, 500, 1000, 1022):
            F = torch.empty(n, 16, device="cuda")
            check(h, spd.spd_learned_features(h, torch.ldexp(A, torch.tensor(k // 2, device="cuda"))
                                              .ldexp(torch.tensor(k - k // 2, device="cuda")).contiguous(), P, 0.1, 0.05, F))
            out[k] = F.cpu().numpy()
        for k, F in out.items():
            assert np.all(np.isfinite(F))
            # s_i into every term, or into the sums: float64 roundings of n terms, then one
            # to float32
            assert np.max(np.abs(F - out[0])) <= 2.0**-23 * max(1.0, np.max(np.abs(out[0]))), k
    finally:
        spd.spd_destroy(h)
