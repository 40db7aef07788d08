"""Calls under a memory cap that leaves room for what they cannot do without: partial
sums that only serve speed are left out, and the call is served."""
import pytest
import torch

import paper_1405_4644_gb300 as spd
import workloads as W
from tests.test_gpu_learned_shapes import loss64

pytestmark = pytest.mark.gpu


def total(*sizes):
    """Bytes of a workspace of these arrays, each on a 256-byte boundary."""
    return sum((s + 255) // 256 * 256 for s in sizes)


@pytest.mark.parametrize("n,p,H", [(1, 1, 8), (33, 3, 16), (700, 17, 130), (1023, 8, 64)])
def test_training_step(n, p, H):
    # vectors of the loss, projections, the preconditioner
    request = total(8 * n, *[8 * n * p] * 7, 8 * 32 * p, 8 * 32 * p, 8 * -(-n // 256) * 32 * p, 8 * (2 * p + 2), 8 * p,
                    8 * n, 8 * 32 * n, 8 * 2048, 4)
    A = W.matern32_torch(W.matern_points(n, 5), 0.2, 0.1, "cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(n + p)
    F = torch.rand(n, 16, device="cuda", generator=g)
    Z = torch.randn(p, n, dtype=torch.float64, device="cuda", generator=g).t()
    T = torch.linalg.solve(A, Z[:, 0]).contiguous()
    h = spd.spd_create(torch.cuda.current_stream())
    try:
        st, net = spd.spd_mlp_create(h, H, 3, False)
        assert st == spd.SPD_OK
        cnt = spd.spd_mlp_params(net)
        params = 0.2 * torch.randn(cnt, device="cuda", generator=g)
        spd.spd_mlp_params(net, inp=params)
        L64, g64 = loss64(torch, params, H, A, F, Z, T, 0.1)
        tol = 2.0 ** -21 * 6 * 100  # as in test_gpu_learned_shapes.test_gradient
        for cap, want in [(request - 1, spd.SPD_ERR_OOM), (request, spd.SPD_OK), (0, spd.SPD_OK)]:
            spd.spd_set_memory_cap(h, cap)
            st, L = spd.spd_mlp_loss_grad(net, A, F, Z, T, 0.1)
            assert st == want, cap
            if st == spd.SPD_OK:
                grad = torch.empty(cnt, device="cuda")
                spd.spd_mlp_params(net, grad=grad)
                assert abs(L - L64) <= tol * abs(L64)
                assert float((grad.double() - g64).norm()) <= tol * float(g64.norm())
        spd.spd_mlp_destroy(net)
    finally:
        spd.spd_destroy(h)
