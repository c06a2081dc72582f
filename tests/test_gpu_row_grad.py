"""The fused gradient row kernel (plans with one bin chunk) of prop_loss_grad
against the oracle: bin groups with dead lanes, one bin, several frames with
and without TV in time, the run of voxels a thread takes not dividing the row,
and a call without a gradient buffer.

Tolerance: the operator at width 8 in FP32 is within 2e-6 (its transforms), the
TV terms d / sqrt(|d|^2 + eps^2) within a few 6e-8 of order-1 values that are
scaled by 1e-2: 5e-6 for the gradient, and for the loss, a sum of squares."""
import numpy as np
import pytest
import torch

import oracle
from helpers import geometry, random_case, rel

pytestmark = pytest.mark.gpu
TOL = 5e-6


@pytest.mark.parametrize("N,Nf,B,L,R,T,tv_t", [
    (16, 1, 3, 4, 16, 1, 0.0),
    (24, 17, 4, 3, 25, 3, 1e-2),   # 16 + 1 bins; T = 3: first, middle and last frame
    (32, 16, 4, 5, 32, 2, 0.0),
    (96, 8, 3, 4, 64, 2, 1e-2),
    (64, 33, 3, 4, 64, 1, 1e-2),   # one frame: TV in time is zero
    (384, 5, 2, 1, 16, 2, 1e-2),   # 24 values a thread
    (512, 3, 2, 1, 16, 1, 0.0),    # 32 values a thread
])
def test_loss_and_gradient(N, Nf, B, L, R, T, tv_t):
    from paper_2311_13177_gb300 import Plan, ReconParams
    c = random_case(N, Nf, B, L, R, T, seed=N + Nf)
    g = geometry(N, L, R, c["theta"], c["delta"], c["blade_frame"], T)
    plan = Plan(N, L, R, c["theta"], c["delta"], c["blade_frame"], T, kb_width=8)
    p = dict(lr=1e-2, tv_xy=1e-2, tv_t=tv_t)
    want, ref = oracle.recon.loss_and_grad(c["V"].astype(np.complex128), c["y"].astype(np.complex128), g,
                                           oracle.ReconParams(iters=1, **p))
    y, V = (torch.from_numpy(c[k]).cuda() for k in ("y", "V"))
    loss, grad = plan.loss_grad(y, ReconParams(iters=1, **p), V)
    plan.destroy()
    assert abs(loss - want) < TOL * abs(want)
    assert rel(grad.cpu().numpy(), ref) < TOL


@pytest.mark.parametrize("N,Nf", [(384, 5), (512, 3)])
def test_update_of_long_rows(N, Nf):
    """Three iterations of the fused update at 24 and 32 values a thread: Adam's
    epsilon of 100, above the gradient's components, makes a step proportional
    to the gradient, whose 5e-6 the volume then has; 1e-5."""
    from paper_2311_13177_gb300 import Plan, ReconParams
    c = random_case(N, Nf, 2, 1, 16, 1, seed=N + Nf)
    g = geometry(N, 1, 16, c["theta"], c["delta"], c["blade_frame"], 1)
    kw = dict(iters=3, lr=1e-1, eps=1e2, tv_xy=5.0, tv_eps=1e-2)
    Vo, tro = oracle.reconstruct(c["y"].astype(np.complex128), g, oracle.ReconParams(**kw))
    plan = Plan(N, 1, 16, c["theta"], c["delta"], c["blade_frame"], 1, kb_width=8)
    V, tr = plan.reconstruct(torch.from_numpy(c["y"]).cuda(), ReconParams(**kw))
    plan.destroy()
    assert rel(V.cpu().numpy(), Vo) < 1e-5
    assert np.max(np.abs(tr - tro) / np.abs(tro)) < 1e-5
