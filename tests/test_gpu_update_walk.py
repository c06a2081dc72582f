"""TV gradient and update of plans with several bin chunks (a thread walks along
x1 with one offset for all arrays) against the oracle: bin counts that do not
divide a block and that exceed it, rows shorter than a walk and not a multiple
of it, a first, middle and last frame; and a volume of more than 4 GB in three
frames, which takes 64-bit offsets.

Tolerances.  Gradient and loss as for the fused kernel (5e-6): the operator at
width 8 in FP32 is within 2e-6, the TV terms within a few 6e-8.  Volume after
three steps: Adam's epsilon of 100, above the gradient's components, makes a
step proportional to the gradient, so its relative error is the gradient's;
1e-5.  Large volume: TV terms d / sqrt(|d|^2 + eps^2) in FP32 (a few 6e-8) with
the data gradient, here below 0.1 of them, rounded to FP32 in both of the
gradients subtracted; 1e-5."""
import numpy as np
import pytest
import torch

import oracle
from helpers import geometry, random_case, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,Nf,T,chunk,tv_t", [
    (16, 33, 3, 16, 5.0),
    (24, 300, 1, 0, 0.0),    # more bins than threads in a block
    (48, 17, 2, 8, 0.0),
    (96, 9, 2, 8, 5.0),
])
def test_gradient_and_update(N, Nf, T, chunk, tv_t):
    from paper_2311_13177_gb300 import Plan, ReconParams
    B, L, R = 4, 3, N
    c = random_case(N, Nf, B, L, R, T, seed=N + Nf)
    g = geometry(N, L, R, c["theta"], c["delta"], c["blade_frame"], T)
    kw = dict(iters=3, lr=1e-1, eps=1e2, tv_xy=5.0, tv_t=tv_t, tv_eps=1e-2)
    want, ref = oracle.recon.loss_and_grad(c["V"].astype(np.complex128), c["y"].astype(np.complex128), g,
                                           oracle.ReconParams(**kw))
    Vo, tro = oracle.reconstruct(c["y"].astype(np.complex128), g, oracle.ReconParams(**kw))
    plan = Plan(N, L, R, c["theta"], c["delta"], c["blade_frame"], T, bin_chunk=chunk, kb_width=8)
    y, V = (torch.from_numpy(c[k]).cuda() for k in ("y", "V"))
    loss, grad = plan.loss_grad(y, ReconParams(**kw), V)
    Vr, tr = plan.reconstruct(y, ReconParams(**kw))
    plan.destroy()
    assert abs(loss - want) < 5e-6 * abs(want)
    assert rel(grad.cpu().numpy(), ref) < 5e-6
    assert rel(Vr.cpu().numpy(), Vo) < 1e-5
    assert np.max(np.abs(tr - tro) / np.abs(tro)) < 1e-5


def test_volume_above_32_bit_offsets():
    from paper_2311_13177_gb300 import Plan, ReconParams
    N, Nf, T, B, L, R = 512, 688, 2, 2, 1, 16
    theta, frames = np.array([0.3, 1.2]), np.array([0, 1], dtype=np.int32)
    plan = Plan(N, L, R, theta, np.linspace(-3, 3, Nf), frames, T, kb_width=8)
    gen = torch.Generator("cuda").manual_seed(5)
    V = torch.view_as_complex(torch.randn((T, N, N, Nf, 2), device="cuda", generator=gen)) * 1e-2
    y = plan.forward(V)
    _, g1 = plan.loss_grad(y, ReconParams(iters=1, tv_xy=1e-2, tv_t=2e-2, tv_eps=1e-3), V)
    _, g0 = plan.loss_grad(y, ReconParams(iters=1, tv_xy=0.0, tv_t=0.0, tv_eps=1e-3), V)
    plan.destroy()
    want = torch.zeros_like(V)
    for axis, weight in ((0, 2e-2), (1, 1e-2), (2, 1e-2)):
        n = V.shape[axis] - 1
        d = V.narrow(axis, 1, n) - V.narrow(axis, 0, n)
        d *= weight / torch.sqrt(d.real ** 2 + d.imag ** 2 + 1e-6)
        want.narrow(axis, 1, n).add_(d)
        want.narrow(axis, 0, n).sub_(d)
    assert float(g0.abs().max()) < 0.1 * float(want.abs().max())
    g1 -= g0
    g1 -= want
    assert float(g1.abs().max()) < 1e-5 * float(want.abs().max())
