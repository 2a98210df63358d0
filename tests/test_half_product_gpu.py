"""Losses by half of the product (rows of H from 3072 entries on): odd and even numbers of blocks of 256, a last block of fewer columns,
few and many layer columns, against fp64 on the GPU."""
import pytest
import torch

from paper_2406_17542_b200 import binding as B
from paper_2406_17542_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_in,d_out,group", [(3072, 130, 0), (3073, 128, 0), (3200, 300, 64), (3328, 257, 0), (3585, 1000, 0), (4100, 129, 4)])
def test_losses_by_half_of_the_product(d_in, d_out, group):
    dev = "cuda:0"
    gen = torch.Generator(dev).manual_seed(d_in)
    X = torch.randn(2000, d_in, generator=gen, device=dev) * torch.randn(d_in, generator=gen, device=dev).exp()
    H = (X.double().T @ X.double()).float()
    H = (torch.tril(H) + torch.tril(H, -1).T).contiguous()
    W = torch.randn(d_in, d_out, generator=gen, device=dev) * 0.02
    grid = B.Grid(3, group, 1, 1.0, 1.0)
    scale, zero, Q, _ = B.cdq_init_rtn(W, grid)
    g = group or d_in
    E = scale.double().repeat_interleave(g, 0) * Q.double() + zero.double().repeat_interleave(g, 0) - W.double()
    want = ((H.double() @ E) * E).sum(0)
    total, got = B.cdq_layer_loss(H, W, grid, scale, zero, Q, per_col=True)
    # The digits of H end 42 bits below a row's power of two, those of a column of E 35 bits below its own, and slice pairs below
    # 2^-63 of the two are left out: at most 2^-42 |e_p| |e_k| row_p + 2^-35 |e_p| |H_pk| col (both counted twice, rounding halves the
    # first) + 12 K 2^-56 row_p col |e_p| (products of two digits of 7 bits).
    row = torch.exp2(torch.frexp(H.abs().amax(1).double())[1].double())
    col = torch.exp2(torch.frexp(E.abs().amax(0))[1].double())
    a = E.abs()
    bound = (2.0 ** -42 * (row @ a) * a.sum(0) + 2.0 ** -34 * (a * H.double().abs().sum(1, keepdim=True)).sum(0) * col
             + 12 * d_in * 2.0 ** -56 * (row @ a) * col + 1e-13 * want.abs())
    assert bool(((got - want).abs() <= bound).all())
    # and far below that where the errors are as random as they are here (3e-12 at most)
    assert float(((got - want) / want).abs().max()) < 1e-11
    assert abs(total - float(want.sum())) <= 1e-12 * float(want.sum())


@pytest.mark.parametrize("base,d_in,d_out,group,given,solved", [("C2", 4096, 512, 128, 1.2e-11, 1.8e-10), ("C3", 3072, 512, 0, 4e-13, 6e-12),
                                                                ("C1", 3073, 130, 0, 8e-12, 1.3e-10)])
def test_precision_of_given_and_solved_codes(base, d_in, d_out, group, given, solved):
    """Relative errors of the column losses against fp64, rms over the columns: round-to-nearest codes, and codes after a descent, whose loss is a
    sum with heavy cancellation that shows every digit lost.  Limits: four times what eight such layers showed (3.0e-12 / 4.5e-11, 9.6e-14 /
    1.4e-12, 2.0e-12 / 3.1e-11; the whole product of truncated slices 5.7e-10 for the solved codes of the first, 2.5e-10 of the last)."""
    dev = "cuda:0"
    X, W = inputs.make_layer(inputs.CONFIGS[base].scaled(d_in=d_in, d_out=d_out, n=2 * d_in, bits=3, group_size=group, seed=50), dev)
    H = torch.zeros(d_in, d_in, dtype=torch.float64, device=dev)
    for rows in X.split(4096):
        H += rows.double().T @ rows.double()
    H = H.float()
    H = (torch.tril(H) + torch.tril(H, -1).T).contiguous()
    grid = B.Grid(3, group, 1, 1.0, 1.0)
    scale, zero, Q, _ = B.cdq_init_rtn(W, grid)
    g = group or d_in
    for limit in (given, solved):
        E = scale.double().repeat_interleave(g, 0) * Q.double() + zero.double().repeat_interleave(g, 0) - W.double()
        want = ((H.double() @ E) * E).sum(0)
        got = B.cdq_layer_loss(H, W, grid, scale, zero, Q, per_col=True)[1]
        assert float((((got - want) / want) ** 2).mean().sqrt()) <= limit
        B.cdq_cd_solve(H, W, grid, scale, zero, Q, 1)


@pytest.mark.parametrize("kind", ["rounding", "triangle", "one NaN", "infinity"])
@pytest.mark.parametrize("d_in,d_out", [(3072, 130), (3333, 300)])
def test_hessians_that_are_not_symmetric_bit_for_bit(d_in, d_out, kind):
    """The loss is e^T H e whatever the class of sizes: of an H whose triangles were rounded apart, of one with a single triangle, of one with
    a NaN whose mirror image is a number (the NaN is left out, the number counts), and of one with infinite entries (left out, like a NaN)."""
    dev = "cuda:0"
    gen = torch.Generator(dev).manual_seed(d_in)
    X = torch.randn(2 * d_in, d_in, generator=gen, device=dev) * torch.randn(d_in, generator=gen, device=dev).exp()
    H = X.double().T @ X.double()
    if kind == "rounding":
        H *= 1 + 1e-6 * torch.randn(d_in, d_in, generator=gen, device=dev).double()
    elif kind == "triangle":
        H = torch.tril(H)
    H = H.float().contiguous()
    there = H.double()
    if kind == "one NaN":
        H[700, 2900] = float("nan")
        there[700, 2900] = 0.0
    if kind == "infinity":
        H[40, 41], H[41, 40], H[2000, 3000] = float("inf"), float("inf"), -float("inf")
        there[40, 41] = there[41, 40] = there[2000, 3000] = 0.0
    W = torch.randn(d_in, d_out, generator=gen, device=dev) * 0.02
    grid = B.Grid(3, 0, 1, 1.0, 1.0)
    scale, zero, Q, _ = B.cdq_init_rtn(W, grid)
    E = scale.double() * Q.double() + zero.double() - W.double()
    want = ((there @ E) * E).sum(0)
    got = B.cdq_layer_loss(H, W, grid, scale, zero, Q, per_col=True)[1]
    # far above the slicing errors (3e-12), far below what one triangle in the place of the other would give (4e-8 and more)
    assert float(((got - want) / want).abs().max()) <= 1e-9
