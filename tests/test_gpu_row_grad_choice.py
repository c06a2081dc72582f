"""prop_loss_grad on both sides of the rule between the fused gradient row kernel
and the separate passes, against the oracle: the shortest and longest fused rows,
a group with one dead lane, few bins over many frames, and lengths that have no
fused kernel.

Tolerance as in test_gpu_row_grad.py: the operator at width 8 within 2e-6, the
TV terms within a few 6e-8 of values that are scaled by 1e-2: 5e-6."""
import numpy as np
import pytest
import torch

import oracle
from helpers import geometry, random_case, rel

pytestmark = pytest.mark.gpu
TOL = 5e-6


@pytest.mark.parametrize("N,Nf,B,L,R,T", [
    (24, 5, 3, 4, 24, 1),      # fused, 2N = 48
    (32, 8, 3, 4, 32, 2),      # fused, 2N = 64
    (384, 16, 2, 1, 16, 1),    # fused, 2N = 768
    (48, 15, 4, 3, 49, 3),     # fused, one dead lane
    (24, 33, 4, 3, 25, 3),     # separate, three groups with 15 dead lanes
    (96, 1, 16, 2, 64, 16),    # separate, one bin
    (512, 2, 2, 1, 16, 2),     # separate, 2N = 1024
])
def test_loss_and_gradient_on_both_sides(N, Nf, B, L, R, T):
    from paper_2311_13177_gb300 import Plan, ReconParams
    c = random_case(N, Nf, B, L, R, T, seed=N + Nf)
    g = geometry(N, L, R, c["theta"], c["delta"], c["blade_frame"], T)
    plan = Plan(N, L, R, c["theta"], c["delta"], c["blade_frame"], T, kb_width=8)
    p = dict(lr=1e-2, tv_xy=1e-2, tv_t=1e-2 if T > 1 else 0.0)
    want, ref = oracle.recon.loss_and_grad(c["V"].astype(np.complex128), c["y"].astype(np.complex128), g,
                                           oracle.ReconParams(iters=1, **p))
    y, V = (torch.from_numpy(c[k]).cuda() for k in ("y", "V"))
    loss, grad = plan.loss_grad(y, ReconParams(iters=1, **p), V)
    plan.destroy()
    assert abs(loss - want) < TOL * abs(want)
    assert rel(grad.cpu().numpy(), ref) < TOL
