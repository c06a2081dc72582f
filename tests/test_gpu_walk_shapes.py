"""Updates whose threads share a row in other ways than the listed sizes do:
bins cut into groups (65, 130), walks cut into unequal last blocks (N = 48 with 6
bins), and the projection model's multi-frame update with and without time
neighbours, against the oracle.

Adam's epsilon of 100 (0.1 in the projection model, whose gradients are smaller)
makes a step a smooth function of the gradient, whose FP32 error is 5e-6: 1e-5."""
import numpy as np
import pytest
import torch

import oracle
from helpers import geometry, random_case, rel
from oracle import projection as pj
from oracle.geometry import make_geometry

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,Nf,T,chunk", [(16, 65, 2, 0), (24, 130, 1, 0), (48, 6, 2, 4)])
def test_chunked_gradient_and_update(N, Nf, T, chunk):
    from paper_2311_13177_gb300 import Plan, ReconParams
    c = random_case(N, Nf, 4, 3, N, T, seed=N + Nf)
    g = geometry(N, 3, N, c["theta"], c["delta"], c["blade_frame"], T)
    kw = dict(iters=3, lr=1e-1, eps=1e2, tv_xy=5.0, tv_t=5.0 if T > 1 else 0.0, tv_eps=1e-2)
    want, ref = oracle.recon.loss_and_grad(c["V"].astype(np.complex128), c["y"].astype(np.complex128), g,
                                           oracle.ReconParams(**kw))
    Vo, tro = oracle.reconstruct(c["y"].astype(np.complex128), g, oracle.ReconParams(**kw))
    plan = Plan(N, 3, N, c["theta"], c["delta"], c["blade_frame"], T, bin_chunk=chunk, kb_width=8)
    y, V = (torch.from_numpy(c[k]).cuda() for k in ("y", "V"))
    loss, grad = plan.loss_grad(y, ReconParams(**kw), V)
    Vr, tr = plan.reconstruct(y, ReconParams(**kw))
    plan.destroy()
    assert abs(loss - want) < 5e-6 * abs(want)
    assert rel(grad.cpu().numpy(), ref) < 5e-6
    assert rel(Vr.cpu().numpy(), Vo) < 1e-5
    assert np.max(np.abs(tr - tro) / np.abs(tro)) < 1e-5


@pytest.mark.parametrize("N,Nf,T,tv_t", [(16, 2, 5, 0.0), (48, 64, 2, 1e-2), (32, 130, 1, 0.0), (48, 6, 1, 0.0),
                                         (16, 33, 4, 1e-2)])
def test_projection_reconstruction(N, Nf, T, tv_t):
    from paper_2311_13177_gb300 import Plan, ProjParams
    B, L, R = 5, 5, N
    rng = np.random.default_rng(N + Nf)
    theta = np.pi * np.arange(B) / B + 0.3
    delta = np.linspace(-4.0, 4.0, Nf)
    frames = (np.arange(B) * T // B).astype(np.int32)
    y = (rng.standard_normal((B, N, N)) + 1j * rng.standard_normal((B, N, N))).astype(np.complex64)
    kw = dict(iters=5, lr=1e-2, eps=1e-1, tv_xy=1e-2, tv_f=1e-2, tv_t=tv_t, l1=1e-3, tv_eps=1e-2)
    Vo, tro = pj.reconstruct(y.astype(np.complex128), None, make_geometry(N, L, R, theta, delta, frames, T),
                             pj.ProjParams(**kw))
    plan = Plan(N, L, R, theta, delta, frames, T, kb_width=8)
    V, tr = plan.proj_reconstruct(torch.from_numpy(y).cuda(), ProjParams(**kw))
    plan.destroy()
    assert rel(V.cpu().numpy(), Vo) < 1e-5
    assert np.max(np.abs(np.asarray(tr) - tro) / np.abs(tro)) < 1e-5
