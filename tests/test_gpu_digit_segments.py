"""The 32-column digit products where a CTA's work items cross its accumulators' limits:
several whole (row block, column group) segments per CTA, and runs of more than 256
items, whose 32-bit sums are flushed in the middle of a segment.  The sums are exact, so
the result has to be that of the 16-column products, bit for bit."""
import pytest
import torch

import paper_1405_4644_gb300 as spd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(300, 3001), (300, 4096), (130, 4090), (20000, 18)])
def test_against_sixteen_columns_at_a_time(n, m):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks, chunks = -(-n // 128), -(-n // 64)
    items = -(-m // 32) * blocks * chunks / sms  # per CTA
    assert items > chunks and (m > 100 or items > 256 + 1)
    g = torch.Generator(device="cuda")
    g.manual_seed(n + m)
    A = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    A *= torch.exp2(torch.randint(-8, 9, (n,), device="cuda", generator=g).double())
    B = torch.randn(m, n, dtype=torch.float64, device="cuda", generator=g).t()
    X = torch.randn(m, n, dtype=torch.float64, device="cuda", generator=g).t()
    R, S = (torch.full((m, n), 7.0, dtype=torch.float64, device="cuda").t() for _ in range(2))
    h = spd.spd_create(torch.cuda.current_stream())
    try:
        assert spd.spd_residual_tc(h, A, B, X, R) == spd.SPD_OK
        for c in range(0, m, 16):
            e = min(m, c + 16)
            assert spd.spd_residual_tc(h, A, B[:, c:e], X[:, c:e], S[:, c:e]) == spd.SPD_OK
    finally:
        spd.spd_destroy(h)
    assert torch.equal(R, S)
