"""The clipping search screens all strengths with a few slice-pair products and forms the accurate loss only
for the strengths within 1 % of a column's smallest screened loss (paper: the grid search over the clipping
strength after Eq. 2).  The screen must never lose the strength the oracle picks from its fp64 loss table:
every column of these layers is compared, on grids whose screen keeps two slices (2, 3 and 4 bits) and on a
finer grid whose screen keeps three (8 bits); a column whose strength differs has to be a near-tie of the
oracle's own table."""
import numpy as np
import pytest
import torch

import oracle
from paper_2406_17542_b200 import binding as B
from paper_2406_17542_b200 import inputs

pytestmark = pytest.mark.gpu

TIE = 1e-7


@pytest.mark.parametrize("base,bits,group,d_in,d_out", [
    ("C2", 2, 128, 2048, 1024),
    ("C4", 3, 128, 2048, 768),
    ("C2", 4, 0, 1536, 512),
    ("C2", 8, 256, 1024, 512),
    ("C2", 2, 128, 3072, 384),      # from 3072 rows on by half of the product
    ("C4", 4, 0, 3328, 300),
    ("C2", 8, 256, 3072, 256),
])
def test_screened_search_picks_the_oracles_strength(base, bits, group, d_in, d_out):
    dev = "cuda:0"
    cfg = inputs.CONFIGS[base].scaled(d_in=d_in, d_out=d_out, n=8192, bits=bits, group_size=group, seed=900 + bits)
    X, W = inputs.make_layer(cfg, device=dev)
    # a few heavy outliers: a clipped weight leaves a residual far above the typical rounding error, which is what the
    # truncating slices of the screen are weakest on
    rng = np.random.default_rng(5)
    rows, cols = rng.integers(0, d_in, 64), rng.integers(0, d_out, 64)
    W[torch.from_numpy(rows).to(dev), torch.from_numpy(cols).to(dev)] *= 6.0
    grid = B.Grid(cfg.bits, cfg.group_size, cfg.n_clip, cfg.clip_lo, cfg.clip_hi)
    H = B.cdq_hessian(X)
    scale, zero, Q, gamma = B.cdq_init_rtn(W, grid, H=H)
    init = oracle.init_rtn(W.cpu(), cfg.bits, cfg.group_size, cfg.n_clip, cfg.clip_lo, cfg.clip_hi, H=H.cpu().numpy(),
                           want_loss_table=True)
    gg = oracle.gamma_grid(cfg.n_clip, cfg.clip_lo, cfg.clip_hi).astype(np.float32)
    got, want = gamma.cpu().numpy(), gg[init["gamma_idx"]]
    differs = np.nonzero(got != want)[0]
    for j in differs:
        t = init["loss_table"][:, j]
        k = int(np.argmin(np.abs(gg - got[j])))
        gap = abs(t[k] - t[init["gamma_idx"][j]]) / t[init["gamma_idx"][j]]
        assert gap <= TIE, (int(j), float(got[j]), float(want[j]), gap)
    same = got == want
    assert np.array_equal(Q.cpu().numpy()[:, same], init["Q"][:, same])
    assert np.array_equal(scale.cpu().numpy()[:, same], init["scale"][:, same])
    print(f"{bits}-bit g={group} {d_in}x{d_out}: strength differs on {len(differs)} of {d_out} columns (near-ties)")


@pytest.mark.parametrize("bits,lo,hi,dominance", [(2, 0.5, 1.0, 500.0), (3, 0.7, 0.8, 80.0), (4, 0.8, 0.9, 200.0), (8, 0.8, 0.9, 2000.0)])
def test_screen_of_rows_that_one_feature_dominates(bits, lo, hi, dominance):
    """Every column against fp64 on the GPU.  One feature is far larger than the others, which all hang together with it, so that its entries
    are the largest of every row of H, but its residual is zero: the loss lies in the small entries.  Strengths close to one another,
    most of them within a few percent of a column's best.  The thirteen-pair losses are good to 1e-6 here."""
    dev, d_in, d_out, n_clip = "cuda:0", 3072, 2048, 20
    lo, hi = float(np.float32(lo)), float(np.float32(hi))   # as the library gets them
    gen = torch.Generator(dev).manual_seed(3)
    z = torch.randn(512, d_in, generator=gen, device=dev)
    sign = torch.randint(0, 2, (d_in,), generator=gen, device=dev).float() * 2 - 1
    X = z + 0.5 * sign * z[:, :1]
    X[:, 0] = dominance * z[:, 0]
    H = (X.double().T @ X.double()).float()
    H = (torch.tril(H) + torch.tril(H, -1).T).contiguous()
    W = torch.randn(d_in, d_out, generator=gen, device=dev) * 0.02
    W[0] = W.amin(0) - 1e-3                       # the zero of the grid: code 0, no residual at any strength
    gamma = B.cdq_init_rtn(W, B.Grid(bits, 0, n_clip, lo, hi), H=H)[3]
    mn, mx, Wd, Hd = W.amin(0).double(), W.amax(0).double(), W.double(), H.double()
    table = []
    for g in oracle.gamma_grid(n_clip, lo, hi):
        a = (float(g) * (mx - mn) / (2 ** bits - 1)).float().double()
        E = a * ((Wd - mn) / a).round().clamp(0, 2 ** bits - 1) + mn - Wd
        table.append(((Hd @ E) * E).sum(0))
    table = torch.stack(table)
    grid = torch.from_numpy(oracle.gamma_grid(n_clip, lo, hi).astype(np.float32)).to(dev)
    chosen = (grid[:, None] == gamma[None, :]).double().argmax(0)
    excess = table.gather(0, chosen[None])[0] / table.amin(0) - 1
    assert float(excess.max()) <= 1e-6


def test_screen_of_a_hessian_that_is_not_positive():
    """A symmetric matrix whose diagonal says nothing about the size of its entries: every column's strength against fp64 all the same."""
    dev, d_in, d_out, n_clip = "cuda:0", 3072, 2048, 8
    gen = torch.Generator(dev).manual_seed(11)
    H = torch.randn(d_in, d_in, generator=gen, device=dev)
    H = (H + H.T).contiguous()
    H.diagonal()[:: 7] = torch.tensor([1e-6, 1e-3, 0.0, -1.0, 30.0], device=dev).repeat(d_in)[: len(range(0, d_in, 7))]
    W = torch.randn(d_in, d_out, generator=gen, device=dev) * 0.02
    gamma = B.cdq_init_rtn(W, B.Grid(3, 0, n_clip, 0.5, 1.0), H=H)[3]
    mn, mx, Wd, Hd = W.amin(0).double(), W.amax(0).double(), W.double(), H.double()
    points = oracle.gamma_grid(n_clip, 0.5, 1.0)
    table = []
    for g in points:
        a = (float(g) * (mx - mn) / 7).float().double()
        E = a * ((Wd - mn) / a).round().clamp(0, 7) + mn - Wd
        table.append(((Hd @ E) * E).sum(0))
    table = torch.stack(table)
    chosen = (torch.from_numpy(points.astype(np.float32)).to(dev)[:, None] == gamma[None, :]).double().argmax(0)
    best = table.amin(0)
    # (losses of both signs: near zero, where the band of a column is narrow, the screen may pass its best strength by)
    wide = best.abs() > 0.02 * table.abs().amax(0)
    excess = ((table.gather(0, chosen[None])[0] - best) / best.abs())[wide]
    assert int(wide.sum()) > d_out // 2 and float(excess.max()) <= 1e-6
