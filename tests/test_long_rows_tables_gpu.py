"""Descent on rows of more than 8192 entries with the tables that fit beside its rows and bounds in shared memory: both, H_ii alone, the group
scales alone, neither; each against the oracle on an H given to both sides."""
import numpy as np
import pytest
import torch

from paper_2406_17542_b200 import binding as B
from paper_2406_17542_b200 import inputs
from util import compare_with_oracle, grid_of

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d_in,g,steps", [(8708, 4, 200), (14336, 128, 300), (14336, 4, 120), (13828, 0, 300), (15364, 4, 120),
                                          (18432, 64, 200), (18432, 4, 80)])
def test_descent_with_the_tables_that_fit(d_in, g, steps):
    cfg = inputs.CONFIGS["C1"].scaled(d_in=d_in, d_out=3, bits=3, group_size=g, x_dtype="bf16", w_dtype="f32", seed=d_in % 97)
    X = inputs.make_x(cfg.scaled(n=768), device=DEV).double()
    H = X.T @ X
    H.diagonal().add_(1e-2 * H.diagonal().mean())
    H = H.float()
    W = inputs.make_w(cfg, device=DEV)
    grid = grid_of(cfg)
    scale, zero, Q0, gamma = B.cdq_init_rtn(W, grid)
    Q = Q0.clone()
    _, _, per = B.cdq_cd_solve_with_loss(H, W, grid, scale, zero, Q, steps, per_col=True)
    assert B.load().cdq_last_device_status() == 0
    compare_with_oracle(cfg, H.cpu().numpy(), H, W, np.arange(3), grid, scale, zero, Q0, Q, gamma, per, steps,
                        label=f"d_in={d_in} g={g} steps={steps}")
