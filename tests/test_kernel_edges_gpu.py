"""Kernels at the edges of their tiles, teams and dispatch rules: odd row lengths, rows that need a padded copy, tiny
budgets, one-bit and eight-bit grids, weights in the middle between two levels."""
import numpy as np
import pytest
import torch

import oracle
from paper_2406_17542_b200 import binding as B
from paper_2406_17542_b200 import inputs
from tests.util import compare_pairs_with_oracle, compare_with_oracle, grid_of

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _layer_h(cfg, rows):
    X = inputs.make_x(cfg.scaled(n=rows), device=DEV).double()
    H = X.T @ X
    H.diagonal().add_(1e-2 * H.diagonal().mean())
    return H.float()


# (d_in, d_out, bits, group, steps): rows just past 8192 entries, odd ones, one level of room, 256 levels, many small
# groups, a full and a ragged team of every width; budgets long enough for thresholds to be drawn anew many times
@pytest.mark.parametrize("d_in,d_out,bits,g,steps", [
    (8196, 5, 1, 0, 400), (8193, 4, 3, 0, 300), (8200, 4, 8, 40, 60), (9216, 4, 2, 4, 400), (8960, 5, 2, 128, 700),
    (14336, 4, 4, 0, 900), (15362, 3, 3, 0, 200), (18432, 3, 3, 128, 500), (8704, 4, 4, 0, 1), (8704, 4, 4, 0, 2),
    # shorter rows that are not a multiple of four: the padded copy, for both of their kernels
    (1023, 9, 3, 0, 900), (1350, 9, 4, 0, 900), (1537, 9, 2, 0, 900), (2050, 9, 3, 0, 900), (5001, 5, 3, 0, 400),
])
def test_descent_at_the_edges(d_in, d_out, bits, g, steps):
    cfg = inputs.CONFIGS["C1"].scaled(d_in=d_in, d_out=d_out, bits=bits, group_size=g, x_dtype="bf16", w_dtype="f32",
                                      seed=700 + d_in % 89)
    H = _layer_h(cfg, 768)
    W = inputs.make_w(cfg, device=DEV)
    W[:, 1] = 0.0123                        # a column without room anywhere
    H[7, :] = 0.0
    H[:, 7] = 0.0                           # a dead feature
    grid = grid_of(cfg)
    scale, zero, Q0, gamma = B.cdq_init_rtn(W, grid)
    Q = Q0.clone()
    stats, loss, per = B.cdq_cd_solve_with_loss(H, W, grid, scale, zero, Q, steps, per_col=True)
    assert B.load().cdq_last_device_status() == 0
    assert stats["steps"] == steps * d_out and stats["committed"] <= steps * (d_out - 1)
    assert torch.equal(Q[:, 1], Q0[:, 1]) and torch.equal(Q[7], Q0[7])
    keep = np.array([c for c in range(d_out) if c != 1])     # (the oracle's audit needs columns that can move)
    compare_with_oracle(cfg, H.cpu().numpy(), H, W, keep, grid, scale, zero, Q0, Q, gamma, per, steps,
                        label=f"d_in={d_in} bits={bits} g={g} steps={steps}")


def test_descent_result_does_not_depend_on_the_other_columns():
    """Columns share a team one after the other, thresholds and watched coordinates included: any subset of the
    columns gives the codes of the whole."""
    cfg = inputs.CONFIGS["C3"].scaled(d_in=8320, d_out=301, bits=3, group_size=64, seed=41)
    H = _layer_h(cfg, 768)
    W = inputs.make_w(cfg, device=DEV)
    grid = grid_of(cfg)
    scale, zero, Q0, _ = B.cdq_init_rtn(W, grid)
    Q = Q0.clone()
    B.cdq_cd_solve(H, W, grid, scale, zero, Q, 0, steps_per_col=600)
    some = torch.arange(3, 301, 13, device=DEV)
    Qs = Q0[:, some].contiguous()
    B.cdq_cd_solve(H, W[:, some].contiguous(), grid, scale[:, some].contiguous(), zero[:, some].contiguous(), Qs, 0,
                   steps_per_col=600)
    assert torch.equal(Qs, Q[:, some])


# (d_in, columns per SM, bits, g): teams of three and of four chunks per thread on either side of their rules, per channel, with group
# scales at a fixed stride (4, 64; 12 on three-chunk teams of 960 and four-chunk teams of 1440 entries) and without one (20)
@pytest.mark.parametrize("d_in,per_sm,bits,g", [
    (769, 6, 3, 0), (1021, 6, 3, 0), (1024, 6, 4, 64), (1024, 5, 3, 0), (772, 6, 3, 4), (960, 6, 3, 12), (960, 6, 2, 20), (840, 6, 8, 24),
    (1153, 8, 3, 0), (1536, 8, 3, 0), (1440, 6, 3, 12), (1440, 6, 3, 20), (1536, 7, 3, 64),
])
def test_descent_of_short_rows_with_many_columns(d_in, per_sm, bits, g):
    d_out = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    cfg = inputs.CONFIGS["C1"].scaled(d_in=d_in, d_out=d_out, bits=bits, group_size=g, w_dtype="f32", seed=800 + d_in % 89)
    H = _layer_h(cfg, 1600)
    W = inputs.make_w(cfg, device=DEV)
    grid = grid_of(cfg)
    scale, zero, Q0, gamma = B.cdq_init_rtn(W, grid)
    Q = Q0.clone()
    _, loss, per = B.cdq_cd_solve_with_loss(H, W, grid, scale, zero, Q, 500, per_col=True)
    assert B.load().cdq_last_device_status() == 0
    some = torch.arange(1, d_out, 37, device=DEV)           # the same columns in a layer of few
    Qs = Q0[:, some].contiguous()
    B.cdq_cd_solve(H, W[:, some].contiguous(), grid, scale[:, some].contiguous(), zero[:, some].contiguous(), Qs, 0,
                   steps_per_col=500)
    assert torch.equal(Qs, Q[:, some])
    compare_with_oracle(cfg, H.cpu().numpy(), H, W, np.array([0, d_out // 2, d_out - 1]), grid, scale, zero, Q0, Q, gamma, per, 500,
                        label=f"d_in={d_in} x {d_out} bits={bits} g={g}")


@pytest.mark.parametrize("d_in,per_sm,bits,g", [(2050, 4, 2, 0), (2050, 3, 2, 0), (2304, 6, 2, 128), (3072, 4, 3, 0), (4096, 4, 2, 64), (4094, 2, 3, 0)])
def test_pairs_on_either_side_of_the_rule_for_their_teams(d_in, per_sm, bits, g):
    """Four pairs per thread for few columns, eight for many, from round-to-nearest codes (where every step moves): the oracle's
    codes, and the same ones from a layer of few columns."""
    d_out = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    cfg = inputs.CONFIGS["C2"].scaled(d_in=d_in, d_out=d_out, bits=bits, group_size=g, n_clip=1, clip_lo=1.0, clip_hi=1.0,
                                      passes=0, seed=820 + d_in % 89)
    H = _layer_h(cfg, 2 * d_in)
    W = inputs.make_w(cfg, device=DEV)
    grid = grid_of(cfg)
    scale, zero, Q0, _ = B.cdq_init_rtn(W, grid)
    Q = Q0.clone()
    B.cdq_bcd_solve(H, W, grid, scale, zero, Q, 2, 40, seed=5)
    _, per = B.cdq_layer_loss(H, W, grid, scale, zero, Q, per_col=True)
    some = torch.arange(2, d_out, 41, device=DEV)
    Qs = Q0[:, some].contiguous()
    B.cdq_bcd_solve(H, W[:, some].contiguous(), grid, scale[:, some].contiguous(), zero[:, some].contiguous(), Qs, 2, 40, seed=5)
    assert B.load().cdq_last_device_status() == 0
    assert torch.equal(Qs, Q[:, some])
    compare_pairs_with_oracle(cfg, H.cpu().numpy(), H, W, np.array([0, 1, d_out - 1]), grid, scale, zero, Q0, Q, per, 40, 5,
                              label=f"d_in={d_in} x {d_out}")


@pytest.mark.parametrize("d_in,at", [(8704, 4096), (8704, 4097), (8704, 8703), (9001, 9000), (4096, 33)])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_a_feature_that_is_not_a_number_shows_in_the_loss(d_in, at, value):
    cfg = inputs.CONFIGS["C3"].scaled(d_in=d_in, d_out=150, bits=3, seed=43)
    H = _layer_h(cfg, 512)
    H[at, :] = value
    H[:, at] = value
    W = inputs.make_w(cfg, device=DEV)
    grid = grid_of(cfg)
    scale, zero, Q0, _ = B.cdq_init_rtn(W, grid)
    Q = Q0.clone()
    stats, loss, per = B.cdq_cd_solve_with_loss(H, W, grid, scale, zero, Q, 40, per_col=True)
    assert B.load().cdq_last_device_status() == 0
    assert not np.isfinite(loss) and not bool(torch.isfinite(per).any())


class _ExactWorkspace:
    """A workspace of exactly the bytes asked for, between bytes of 0xFF (NaN as floats and doubles) that the library has
    no business with."""
    GUARD = 1 << 20      # rows of padding are at most 3 x 18432 floats

    def get(self, nbytes, device):
        self.need = nbytes
        self.buf = torch.full((nbytes + 2 * self.GUARD,), 0xFF, dtype=torch.uint8, device=device)
        return self.buf.data_ptr() + self.GUARD, nbytes

    def guards_intact(self):
        return bool((self.buf[:self.GUARD] == 0xFF).all()) and bool((self.buf[self.GUARD + self.need:] == 0xFF).all())


# (few columns: the padded copy of H is the last block; 200 columns of 301: in the place of the residual; the rest: of the slices)
@pytest.mark.parametrize("d_in,d_out", [(1029, 3), (5001, 3), (8193, 3), (8194, 3), (8195, 3), (9001, 3), (18431, 3), (301, 200),
                                        (1351, 300), (8202, 130)])
def test_padding_of_odd_rows_takes_nothing_from_behind_the_workspace(d_in, d_out):
    """The padding coordinates of an odd layer have no row in H.  Their gradients lie in the workspace (behind the residual,
    [columns, d_in rounded up to 4] doubles) and stay zero whatever follows the workspace in memory."""
    cfg = inputs.CONFIGS["C3"].scaled(d_in=d_in, d_out=d_out, bits=3, seed=44)
    H = _layer_h(cfg, 256)
    W = inputs.make_w(cfg, device=DEV)
    grid = grid_of(cfg)
    scale, zero, Q, _ = B.cdq_init_rtn(W, grid)
    ws = _ExactWorkspace()
    _, loss, per = B.cdq_cd_solve_with_loss(H, W, grid, scale, zero, Q, 30, per_col=True, ws=ws)
    assert B.load().cdq_last_device_status() == 0
    assert np.isfinite(loss) and bool(torch.isfinite(per).all()) and ws.guards_intact()
    ldg = (d_in + 3) // 4 * 4
    off = ws.GUARD + (8 * d_in * d_out + 255) // 256 * 256
    G = ws.buf[off:off + 8 * d_out * ldg].view(torch.float64).view(d_out, ldg)
    assert bool((G[:, d_in:] == 0).all()) and bool(torch.isfinite(G).all())
    want, cols = B.cdq_layer_loss(H, W, grid, scale, zero, Q, per_col=True)
    assert abs(loss - want) <= 1e-9 * want and bool(((per - cols).abs() <= 1e-9 * cols).all())


def test_pairs_need_no_room_for_padded_rows():
    """Pairs read H as it is: a workspace for the descent without the padded copy is enough (1026 entries: 4.2 MB)."""
    cfg = inputs.CONFIGS["C3"].scaled(d_in=1026, d_out=8, bits=3, seed=45)
    H = _layer_h(cfg, 1100)
    W = inputs.make_w(cfg, device=DEV)
    grid = grid_of(cfg)
    scale, zero, Q, _ = B.cdq_init_rtn(W, grid)
    Q2 = Q.clone()
    want = B.cdq_bcd_solve(H, W, grid, scale, zero, Q, 2, 16, seed=3)

    class Smaller(_ExactWorkspace):   # less the padded copy, plus the pairs of 16 steps (16 bytes each)
        def get(self, nbytes, device):
            return super().get(nbytes - (4 * 1026 * 1028) // 256 * 256 + 16 * 16 * 1026, device)

    ws = Smaller()
    got = B.cdq_bcd_solve(H, W, grid, scale, zero, Q2, 2, 16, seed=3, ws=ws)
    assert torch.equal(Q, Q2) and got["committed"] == want["committed"] and ws.guards_intact()


@pytest.mark.parametrize("d_in", [8704, 8705])
@pytest.mark.parametrize("i,k", [(4096, 17), (4097, 33), (8703, 8702), (6, 5)])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
def test_an_entry_off_the_diagonal_that_is_not_a_number_shows_in_the_loss(d_in, i, k, value):
    """At even and odd places of a row; only the two features at its ends are kept from moving."""
    cfg = inputs.CONFIGS["C3"].scaled(d_in=d_in, d_out=40, bits=3, seed=47)
    H = _layer_h(cfg, 512)
    H[i, k] = H[k, i] = value
    W = inputs.make_w(cfg, device=DEV)
    grid = grid_of(cfg)
    scale, zero, Q0, _ = B.cdq_init_rtn(W, grid)
    Q = Q0.clone()
    _, loss, per = B.cdq_cd_solve_with_loss(H, W, grid, scale, zero, Q, 40, per_col=True)
    assert B.load().cdq_last_device_status() == 0
    assert not np.isfinite(loss) and not bool(torch.isfinite(per).any())
    assert torch.equal(Q[i], Q0[i]) and torch.equal(Q[k], Q0[k])


def _float_of_bits(bits):
    return torch.from_numpy(np.array([bits], dtype=np.uint32).view(np.int32)).to(DEV).view(torch.float32)


# (layers whose gradient comes from the int8 product, for each of the descent's kernels, and from both fp64 products)
@pytest.mark.parametrize("d_in,d_out", [(512, 1600), (1024, 600), (2048, 128), (8704, 128), (256, 128), (301, 400), (256, 6000)])
@pytest.mark.parametrize("bits", [0x7FC00000, 0x7FFFFFFF, 0xFFFFFFFF, 0x7F800001])
def test_a_nan_is_left_out_of_the_gradient_whatever_its_payload(d_in, d_out, bits):
    """0x7FFFFFFF is the NaN that CUDA's arithmetic makes, 0x7FC00000 that of a Python literal.  A NaN weight takes code 0 and
    leaves its column as one with the zero of the grid there, a NaN feature of H its layer as one without the feature; the
    losses of the descent show both."""
    cfg = inputs.CONFIGS["C3"].scaled(d_in=d_in, d_out=d_out, bits=3, seed=46)
    H = _layer_h(cfg, 768)
    W = inputs.make_w(cfg, device=DEV)
    grid = grid_of(cfg)
    T = min(d_in, 600)
    nan = _float_of_bits(bits)

    def solve(Hs, Ws):
        scale, zero, Q, _ = B.cdq_init_rtn(Ws, grid)
        _, loss, per = B.cdq_cd_solve_with_loss(Hs, Ws, grid, scale, zero, Q, T, per_col=True)
        assert B.load().cdq_last_device_status() == 0
        return Q, per

    Wn, Wz = W.clone(), W.clone()
    Wn[5, 3:4] = nan
    Wz[5, 3] = torch.cat([W[:5, 3], W[6:, 3]]).min()
    Q, per = solve(H, Wn)
    Qz, perz = solve(H, Wz)
    assert torch.equal(Q, Qz)
    assert bool(per[3].isnan()) and torch.equal(per[:3], perz[:3]) and torch.equal(per[4:], perz[4:])
    Hn, Hz = H.clone(), H.clone()
    Hn[7, :], Hn[:, 7] = nan.expand(d_in), nan.expand(d_in)
    Hz[7, :], Hz[:, 7] = 0.0, 0.0
    Q, per = solve(Hn, W)
    Qz, _ = solve(Hz, W)
    assert torch.equal(Q, Qz) and bool(per.isnan().all())
    scale, zero, Q, _ = B.cdq_init_rtn(W, grid)
    loss, lossz = (B.cdq_layer_loss(Hs, W, grid, scale, zero, Q) for Hs in (Hn, Hz))
    assert loss == lossz and np.isfinite(loss)


@pytest.mark.parametrize("d_in,width", [(256, 256), (257, 264), (319, 320), (384, 392), (641, 648), (1158, 1160), (1283, 1288)])
def test_hessian_pieces_and_mirror(d_in, width):
    """bf16 rows with a stride longer than d_in through the tensor-core kernel: every entry against fp64 (3e-5 of
    sqrt(H_ii H_jj), the bar of the tensor-core path for up to 4096 rows), symmetric bit for bit, accumulated too."""
    g = torch.Generator(device=DEV).manual_seed(d_in)
    X = torch.randn((1536, width), generator=g, device=DEV).bfloat16()
    Xv = X[:, :d_in]
    H = B.cdq_hessian(Xv)
    D = Xv.double()
    want = D.T @ D
    norm = torch.sqrt(torch.outer(want.diagonal(), want.diagonal()))
    assert float(((H.double() - want).abs() / norm).max()) <= 3e-5
    assert torch.equal(H, H.T.contiguous())
    H2 = B.cdq_hessian(Xv, accumulate=True, out=H.clone())
    assert torch.equal(H2, 2 * H)           # the second sum is the same, and doubling is exact


@pytest.mark.parametrize("d_in", [1, 15, 16, 17, 33, 255, 511, 512, 513, 577, 1023, 1024, 1025, 1091])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_hessian_on_the_cuda_cores(d_in, dtype):
    """Every tile size with odd edges, rows not a multiple of a stage, accumulated: fp64 sums rounded once to fp32,
    so within half a unit in the last place (6e-8) of the exact sum plus the fp64 sum's own 2e-13."""
    g = torch.Generator(device=DEV).manual_seed(d_in)
    X = torch.randn((203, d_in + 3), generator=g, device=DEV).to(dtype)[:, :d_in]
    H = B.cdq_hessian(X)
    D = X.double()
    want = D.T @ D
    norm = torch.sqrt(torch.outer(want.diagonal(), want.diagonal()))
    assert float(((H.double() - want).abs() / norm).max()) <= 6.1e-8
    assert torch.equal(H, H.T.contiguous())
    H2 = B.cdq_hessian(X, accumulate=True, out=H.clone())
    assert float(((H2.double() - 2 * want).abs() / norm).max()) <= 2.5e-7


@pytest.mark.parametrize("d_in,d_out,bits,g,dtype", [
    (64, 8, 8, 16, "f32"), (48, 5, 3, 0, "f32"), (520, 1028, 4, 130, "bf16"), (1024, 1024, 8, 0, "f32"), (1000, 516, 2, 8, "f32"),
])
def test_codes_of_weights_between_two_levels(d_in, d_out, bits, g, dtype):
    """Weights in the middle between two levels and one fp32 neighbour to either side: bit for bit the oracle's codes,
    in the one-column and the four-column kernel."""
    rng = np.random.default_rng(d_in + bits)
    gg = g or d_in
    L = 2 ** bits - 1
    W = rng.standard_normal((d_in, d_out)).astype(np.float32) * 0.02
    for t in range(d_in // gg):
        blk = W[t * gg:(t + 1) * gg]
        lo, hi = blk.min(0).astype(np.float64), blk.max(0).astype(np.float64)
        a = (hi - lo) / L
        k = rng.integers(0, L, blk.shape)
        mid = (lo + a * (k + 0.5)).astype(np.float32)
        mid = np.where(rng.random(blk.shape) < 0.3, np.nextafter(mid, np.float32(1)), mid)
        mid = np.where(rng.random(blk.shape) < 0.3, np.nextafter(mid, np.float32(-1)), mid)
        keep = (blk == blk.min(0)) | (blk == blk.max(0))
        W[t * gg:(t + 1) * gg] = np.where(keep, blk, mid)
    Wt = torch.from_numpy(W)
    if dtype == "bf16":
        Wt = Wt.bfloat16()
    want = oracle.init_rtn(Wt, bits, g, 1, 1.0, 1.0)
    scale, zero, Q, _ = B.cdq_init_rtn(Wt.to(DEV), B.Grid(bits, g))
    assert np.array_equal(scale.cpu().numpy(), want["scale"]) and np.array_equal(zero.cpu().numpy(), want["zero"])
    assert np.array_equal(Q.cpu().numpy(), want["Q"])


@pytest.mark.parametrize("d_in,d_out,bits,g,dtype", [
    (64, 32, 2, 0, "f32"), (64, 32, 3, 16, "f32"), (96, 33, 8, 0, "bf16"), (4096, 1024, 4, 0, "f32"),
])
def test_codes_of_groups_that_span_more_than_the_largest_float(d_in, d_out, bits, g, dtype):
    """w - b overflows in fp32 (the scale does not, from two bits on): the oracle's codes all the same, in the codes and in the
    residuals of the clipping search."""
    rng = np.random.default_rng(bits)
    Wt = torch.from_numpy((3e38 * (2 * rng.random((d_in, d_out)) - 1)).astype(np.float32))
    if dtype == "bf16":
        Wt = Wt.bfloat16()
    want = oracle.init_rtn(Wt, bits, g, 1, 1.0, 1.0)
    scale, zero, Q, _ = B.cdq_init_rtn(Wt.to(DEV), B.Grid(bits, g))
    assert np.array_equal(scale.cpu().numpy(), want["scale"]) and np.array_equal(zero.cpu().numpy(), want["zero"])
    assert np.array_equal(Q.cpu().numpy(), want["Q"])
    if d_in > 96:
        return
    X = torch.from_numpy(rng.standard_normal((4 * d_in, d_in)).astype(np.float32))
    H = (X.double().T @ X.double()).float()
    # (strengths from 0.5: the library takes the ends of the grid as floats, the oracle as doubles, and 0.6 is another number as each)
    want = oracle.init_rtn(Wt, bits, g, 5, 0.5, 1.0, H=H.numpy())
    scale, zero, Q, gamma = B.cdq_init_rtn(Wt.to(DEV), B.Grid(bits, g, 5, 0.5, 1.0), H=H.to(DEV))
    assert np.array_equal(gamma.cpu().numpy(), oracle.gamma_grid(5, 0.5, 1.0).astype(np.float32)[want["gamma_idx"]])
    assert np.array_equal(scale.cpu().numpy(), want["scale"]) and np.array_equal(Q.cpu().numpy(), want["Q"])
