"""Plans whose spread lists outgrow a shared-memory stage while the bin stride
has kernels of its own: the grouped lists give way to cell lists over the whole
grid (staged, and with more blades gathered from global memory), beside either
interpolation, also where the samples reach less than half of the grid.

Tolerance: width 8's own error is 5e-8 and the transforms are 14 radix-2 stages
of a few 6e-8 roundings, so 2e-6; a gradient put together from the two
operators differs from them by their own rounding only, 2e-6 as well."""
import numpy as np
import pytest
import torch

import oracle
from helpers import geometry, random_case, rel

pytestmark = pytest.mark.gpu
TOL = 2e-6


@pytest.mark.parametrize("N,Nf,B,L,R", [
    (64, 16, 130, 6, 64),     # cell lists, staged
    (64, 16, 130, 8, 24),     # a short readout: the middle of the grid only
    (64, 8, 1400, 2, 24),     # cell lists in global memory
    (32, 64, 200, 6, 24),     # bin stride 64
])
def test_cell_lists_beside_the_stride_kernels(N, Nf, B, L, R):
    from paper_2311_13177_gb300 import Plan, ReconParams
    c = random_case(N, Nf, B, L, R, 1, seed=N + B)
    g = geometry(N, L, R, c["theta"], c["delta"], c["blade_frame"], 1)
    plan = Plan(N, L, R, c["theta"], c["delta"], c["blade_frame"], 1, kb_width=8)
    V, y = (torch.from_numpy(c[k]).cuda() for k in ("V", "y"))
    rng = np.random.default_rng(B)
    bad = torch.full_like(V, float("nan"))
    plan.forward(bad)                      # a grid full of NaN
    Va = plan.adjoint(y)
    plan.forward(bad)
    Ay = plan.forward(V)
    r = Ay - y
    want = 2 * plan.adjoint(r)
    loss, grad = plan.loss_grad(y, ReconParams(iters=1, tv_xy=0.0), V)
    again = plan.adjoint(y)
    plan.destroy()
    s = rng.choice(Ay.numel(), 1024, replace=False)
    assert rel(Ay.cpu().numpy().reshape(-1)[s], oracle.forward_at(c["V"].astype(np.complex128), g, s)) < TOL
    q = rng.choice(Va.numel(), 256, replace=False)
    assert rel(Va.cpu().numpy().reshape(-1)[q], oracle.adjoint_at(c["y"].astype(np.complex128), g, q)) < TOL
    assert torch.equal(again, Va)
    assert rel(grad.cpu().numpy(), want.cpu().numpy()) < TOL
    d = float((r.real.double() ** 2 + r.imag.double() ** 2).sum())
    assert abs(loss - d) < TOL * d
