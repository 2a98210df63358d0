"""Hessians whose tiles the product itself adds to H (no K splits): odd widths, a last tile row and column of a few features, rows of H off
16-byte boundaries, several chunks of calibration rows per tile, accumulation."""
import pytest
import torch

from paper_2406_17542_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n,d_in,width", [(1536, 4224, 4224), (1500, 4354, 4360), (1536, 4609, 4616), (1000, 4100, 4104), (16600, 4100, 4104)])
def test_tiles_added_to_the_hessian(n, d_in, width):
    """Every entry against fp64 (3e-5 of sqrt(H_ii H_jj) up to 4096 rows; the accumulators' error grows with the rows in them: 1e-4 up to 16384),
    symmetric bit for bit, added to what was there."""
    g = torch.Generator(device=DEV).manual_seed(d_in)
    X = torch.randn((n, width), generator=g, device=DEV).bfloat16()[:, :d_in]
    H = B.cdq_hessian(X)
    D = X.double()
    want = D.T @ D
    norm = torch.sqrt(torch.outer(want.diagonal(), want.diagonal()))
    bar = 3e-5 if n <= 4096 else 1e-4
    assert float(((H.double() - want).abs() / norm).max()) <= bar
    assert torch.equal(H, H.T.contiguous())
    assert torch.equal(B.cdq_hessian(X, accumulate=True, out=H.clone()), 2 * H)   # the second sum is the same, and doubling is exact
    other = torch.randn((d_in, d_in), generator=g, device=DEV)
    other = (other + other.T).contiguous()
    assert torch.equal(B.cdq_hessian(X, accumulate=True, out=other.clone()), H + other)
