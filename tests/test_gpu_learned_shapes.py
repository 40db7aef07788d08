"""The training step where its splits end: rows, probes and widths around the
slices of the weight gradients, the row chunks and the column blocks of the float64
products, against the same network in float64 by torch's own differentiation."""
import numpy as np
import pytest

import paper_1405_4644_gb300 as spd
import workloads as W

pytestmark = pytest.mark.gpu

from tests.gpu_util import check, dev_sym  # noqa: E402


@pytest.fixture(scope="module")
def h():
    import torch
    hh = spd.spd_create(torch.cuda.current_stream())
    yield hh
    spd.spd_destroy(hh)


def loss64(torch, params, H, A, F, Z, T, w):
    p = params.double().requires_grad_()
    cut = np.cumsum([0, 16 * H, H, H * H, H, 33 * H, 33])
    W1, b1, W2, b2, W3, b3 = (p[int(i):int(j)] for i, j in zip(cut, cut[1:]))
    silu = torch.nn.functional.silu
    O = silu(silu(F.double() @ W1.view(H, 16).T + b1) @ W2.view(H, H).T + b2) @ W3.view(33, H).T + b3
    s = A.diagonal().rsqrt()
    M = torch.linalg.inv(torch.diag(torch.nn.functional.softplus(O[:, 0]) + 1e-3) + O[:, 1:] @ O[:, 1:].T)
    Y = s[:, None] * (M @ (s[:, None] * Z))
    E = A @ Y - Z
    L = ((E ** 2).sum(0) / (Z ** 2).sum(0)).mean() + w * ((Y[:, 0] - T) ** 2).sum() / (T ** 2).sum()
    return float(L), torch.autograd.grad(L, p)[0]


@pytest.mark.parametrize("n,p,H", [(1, 1, 8), (31, 2, 16), (32, 1, 9), (33, 3, 16), (127, 4, 24), (128, 5, 64), (129, 8, 65),
                                   (257, 9, 33), (600, 16, 40), (700, 17, 130), (1023, 33, 64), (4100, 2, 16)])
def test_gradient(h, n, p, H):
    import torch
    A = W.matern32_torch(W.matern_points(n, 5), 0.2, 0.1, "cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(n + p)
    F = torch.rand(n, 16, device="cuda", generator=g)
    Z = torch.randn(p, n, dtype=torch.float64, device="cuda", generator=g).t()
    T = torch.linalg.solve(A, Z[:, 0]).contiguous()
    st, net = spd.spd_mlp_create(h, H, 3, False)
    check(h, st)
    cnt = spd.spd_mlp_params(net)
    params = 0.2 * torch.randn(cnt, device="cuda", generator=g)
    spd.spd_mlp_params(net, inp=params)
    st, L = spd.spd_mlp_loss_grad(net, A, F, Z, T, 0.1)
    check(h, st)
    grad = torch.empty(cnt, device="cuda")
    spd.spd_mlp_params(net, grad=grad)
    spd.spd_mlp_destroy(net)
    L64, g64 = loss64(torch, params, H, A, F, Z, T, 0.1)
    # a float32 network (exponentials to about 2^-21) behind a float64 loss: 2^-21
    # times the length of the chain (three layers forward and back) and the loss's
    # conditioning, taken as 100
    tol = 2.0 ** -21 * 6 * 100
    assert abs(L - L64) <= tol * abs(L64)
    assert float((grad.double() - g64).norm()) <= tol * float(g64.norm())


@pytest.mark.parametrize("n", [1, 2, 31, 127, 129, 513])
def test_features(h, n):
    import torch
    from oracle import learned as ol
    pts = W.matern_points(n, 2)
    A = W.matern32_torch(pts, 0.1, 0.05, "cuda")
    F = torch.empty(n, 16, device="cuda")
    check(h, spd.spd_learned_features(h, A, torch.from_numpy(pts).to("cuda"), 0.1, 0.05, F))
    want = ol.features(A.cpu().numpy(), pts, 0.1, 0.05)
    # one rounding to float32, float64 sums
    assert np.max(np.abs(F.cpu().numpy() - want)) <= 2.0 ** -23 * max(1.0, np.max(np.abs(want)))
