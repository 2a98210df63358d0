"""GPU parity of cdq_init_owc_cd (paper: Algorithm 3) against the fp64 CPU oracle.

Bars: in the fp64 verification mode the chosen grid indices, scales, zeros, codes, number of
changes and per-column losses are bit-exact; in the production mode (same arithmetic, other
summation order) at least 99 % of the (group, column) strengths agree, the columns whose strengths
all agree have identical codes, and the layer loss is within 1e-6 relative."""
import numpy as np
import pytest
import torch

import oracle
from paper_2406_17542_b200 import binding as B
from paper_2406_17542_b200 import inputs

pytestmark = pytest.mark.gpu

CASES = [  # d_in, d_out, n, bits, g, n_clip, steps
    (64, 20, 300, 3, 16, 6, 0),
    (96, 33, 400, 2, 32, 5, 2),
    (48, 7, 200, 4, 0, 8, 1),       # one group per column: one step is the OWC grid search
    (256, 40, 1024, 2, 64, 20, 0),
    (36, 9, 150, 3, 12, 4, 50),     # run to convergence
]


@pytest.mark.parametrize("d_in,d_out,n,bits,g,n_clip,steps", CASES)
@pytest.mark.parametrize("mode", ["verify", "fast"])
def test_owc_cd_matches_oracle(d_in, d_out, n, bits, g, n_clip, steps, mode):
    cfg = inputs.CONFIGS["C2"].scaled(d_in=d_in, d_out=d_out, n=n, bits=bits, group_size=g, n_clip=n_clip,
                                      clip_lo=0.5, clip_hi=1.0, seed=500 + d_in)
    X, W = inputs.make_layer(cfg)
    _, H32 = oracle.hessian(X)
    ng = d_in // (g or d_in)
    ref = oracle.owc_cd(H32, W, bits, g, n_clip, 0.5, 1.0, steps if steps > 0 else ng)
    grid = B.Grid(bits, g, n_clip, 0.5, 1.0)
    Hd = torch.from_numpy(H32).cuda()
    scale, zero, Q, gamma, stats = B.cdq_init_owc_cd(W.cuda(), grid, Hd, steps=steps, mode=mode)
    torch.cuda.synchronize()
    gam_ref = oracle.gamma_grid(n_clip, 0.5, 1.0)[ref["gamma_idx"]].astype(np.float32)
    got_gamma = gamma.cpu().numpy()
    if mode == "verify":
        assert np.array_equal(got_gamma, gam_ref)
        assert np.array_equal(scale.cpu().numpy(), ref["scale"])
        assert np.array_equal(zero.cpu().numpy(), ref["zero"])
        assert np.array_equal(Q.cpu().numpy(), ref["Q"])
        assert stats["moves"] == int(ref["moves"].sum())
        # totals are ascending sums of the per-column values on both sides
        assert stats["loss_before"] == float(np.cumsum(ref["loss_before"])[-1])
        assert stats["loss_after"] == float(np.cumsum(ref["loss_after"])[-1])
    else:
        same = got_gamma == gam_ref
        assert same.mean() >= 0.99, same.mean()
        cols = np.nonzero(same.all(axis=0))[0]
        assert np.array_equal(Q.cpu().numpy()[:, cols], ref["Q"][:, cols])
        assert np.array_equal(scale.cpu().numpy()[:, cols], ref["scale"][:, cols])
        np.testing.assert_allclose(stats["loss_after"], ref["loss_after"].sum(), rtol=1e-6)
        np.testing.assert_allclose(stats["loss_before"], ref["loss_before"].sum(), rtol=1e-9)
    # the reported loss is the loss of what was emitted
    loss = B.cdq_layer_loss(Hd, W.cuda(), B.Grid(bits, g), scale, zero, Q, mode="verify")
    np.testing.assert_allclose(stats["loss_after"], loss, rtol=1e-9)
    assert stats["loss_after"] <= stats["loss_before"]


@pytest.mark.parametrize("d_in,d_out,n,bits,g,n_clip,steps", [
    # production kernels on either side of their limits: groups of 40 and 512 coordinates, two per strength; odd ones, whose codes and
    # gradients lie off the vectors' boundaries; 32 and 33 strengths; two strengths; eight bits
    (120, 9, 500, 3, 40, 21, 0), (120, 9, 500, 3, 40, 22, 0), (117, 9, 500, 3, 39, 6, 0), (205, 11, 700, 2, 41, 5, 0),
    (512, 5, 900, 3, 512, 6, 3), (130, 7, 600, 4, 65, 32, 0), (130, 7, 600, 4, 65, 33, 0), (342, 6, 900, 8, 57, 2, 0),
])
def test_owc_cd_matches_oracle_at_the_limits_of_its_kernels(d_in, d_out, n, bits, g, n_clip, steps):
    test_owc_cd_matches_oracle(d_in, d_out, n, bits, g, n_clip, steps, "fast")


def test_owc_cd_then_descent_never_worse_than_owc_then_descent_start():
    """Per-group strengths start the descent at or below the loss of the one-strength-per-column search."""
    cfg = inputs.CONFIGS["C2"].scaled(d_in=512, d_out=160, n=2048, seed=9)
    X, W = inputs.make_layer(cfg, device="cuda:0")
    grid = B.Grid(cfg.bits, cfg.group_size, cfg.n_clip, cfg.clip_lo, cfg.clip_hi)
    H = B.cdq_hessian(X)
    s1, z1, Q1, _ = B.cdq_init_rtn(W, grid, H=H)
    l1 = B.cdq_layer_loss(H, W, grid, s1, z1, Q1)
    s2, z2, Q2, _, st = B.cdq_init_owc_cd(W, grid, H, steps=50 * (cfg.d_in // cfg.group_size))
    l2 = B.cdq_layer_loss(H, W, grid, s2, z2, Q2)
    np.testing.assert_allclose(st["loss_after"], l2, rtol=1e-6)
    assert l2 <= st["loss_before"]
    print("OWC loss", l1, "OWC-CD loss", l2, "moves", st["moves"])
