"""Grid and codes of small groups by one block each (many groups, no clipping search) against the general path, which pieces of the same
layer with few groups take: bit for bit, with weights in the middle between two levels, constant groups, infinities and NaN."""
import pytest
import torch

from paper_2406_17542_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("g,ng,d_out,bits", [(4, 200, 500, 3), (20, 150, 516, 2), (32, 148, 512, 4), (36, 150, 640, 3), (64, 160, 492, 8),
                                             (100, 150, 508, 1), (128, 149, 512, 3)])
def test_codes_of_a_group_per_block(g, ng, d_out, bits, dtype):
    gen = torch.Generator(DEV).manual_seed(g + bits)
    W = torch.randn(g * ng, d_out, generator=gen, device=DEV) * 0.02
    L = 2 ** bits - 1
    W[:g, :8] = torch.arange(g, device=DEV).float()[:, None] % (2 * L + 1) * 0.5     # every level and every middle
    W[0, :8], W[1, :8] = 0.0, float(L)
    W[g:2 * g, 9] = 0.25                                                            # a constant group
    W[2 * g, 11], W[3 * g + 1, 12], W[4 * g + 2, 13] = float("nan"), float("inf"), -float("inf")
    W[5 * g:6 * g, 14] = float("nan")
    W[6 * g:7 * g, 15] *= 1e-38
    W = W.to(dtype)
    grid = B.Grid(bits, g, 1, 1.0, 1.0)
    scale, zero, Q, gamma = B.cdq_init_rtn(W, grid)
    per = max(1, 500 // ((d_out + 127) // 128))          # groups of a piece: fewer blocks than the rule asks for
    assert (d_out + 127) // 128 * ng >= 592 > (d_out + 127) // 128 * per
    for t in range(0, ng, per):
        s, z, q, _ = B.cdq_init_rtn(W[t * g:(t + per) * g].contiguous(), grid)
        assert torch.equal(q, Q[t * g:(t + per) * g])
        for a, b in ((s, scale[t:t + per]), (z, zero[t:t + per])):
            assert torch.equal(torch.isnan(a), torch.isnan(b)) and torch.equal(a.nan_to_num(1.5), b.nan_to_num(1.5))
