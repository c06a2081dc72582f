"""Projection-model reconstruction against the oracle where the update's thread
layout and the fused column passes can go wrong: one bin, bin counts that do
not divide a block and that exceed it, a first, middle and last frame, shifts
of more than half the image, the data off the mask NaN (they are not used).

Adam's epsilon of 0.1 makes a step a smooth function of the gradient, so that
the volume carries the gradient's FP32 error (1e-6 of it: 2 log2(N^2) roundings of
6e-8 in the transforms) and not the sign of components near zero: 1e-5 asked."""
import numpy as np
import pytest
import torch

from helpers import rel
from oracle import projection as pj
from oracle.geometry import make_geometry

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,Nf,T,span,with_image", [
    (16, 1, 1, 3.0, False),
    (48, 33, 3, 4.0, True),
    (32, 8, 2, 20.0, False),   # shifts beyond half the image
    (16, 300, 1, 4.0, False),  # more bins than threads in a block
    (48, 16, 1, 4.0, True),
])
def test_reconstruction(N, Nf, T, span, with_image):
    from paper_2311_13177_gb300 import Plan, ProjParams
    B, L, R = 3, 5, N
    rng = np.random.default_rng(N + Nf)
    theta = np.pi * np.arange(B) / B + 0.3
    delta = np.linspace(-span, span, Nf) if Nf > 1 else np.array([1.7])
    frames = (np.arange(B) * T // B).astype(np.int32)
    g = make_geometry(N, L, R, theta, delta, frames, T)
    cplx = lambda *s: (rng.standard_normal(s) + 1j * rng.standard_normal(s)).astype(np.complex64)  # noqa: E731
    y = cplx(B, N, N)
    img = cplx(B, N, N) if with_image else None
    kw = dict(iters=4, lr=1e-2, eps=1e-1, tv_xy=1e-2, tv_f=1e-2, tv_t=1e-2 if T > 1 else 0.0, l1=1e-3, tv_eps=1e-2)
    Vo, tro = pj.reconstruct(y.astype(np.complex128), None if img is None else img.astype(np.complex128), g,
                             pj.ProjParams(**kw))
    mask = np.stack([pj.blade_mask(N, theta[b], L, R) for b in range(B)])
    y = np.where(mask, y, np.complex64(complex("nan"))).astype(np.complex64)
    plan = Plan(N, L, R, theta, delta, frames, T)
    V, tr = plan.proj_reconstruct(torch.from_numpy(y).cuda(), ProjParams(**kw),
                                  img=None if img is None else torch.from_numpy(img).cuda())
    plan.destroy()
    assert rel(V.cpu().numpy(), Vo) < 1e-5
    assert np.max(np.abs(tr - tro) / np.abs(tro)) < 1e-5


def test_volume_above_32_bit_offsets():
    """Without data weights and spectral terms each bin is a problem of its own:
    the bins of a volume of more than 4 GB in three frames, which repeat those of
    a small one, get the same updates (the same operations; a few roundings of
    6e-8 of the values asked)."""
    from paper_2311_13177_gb300 import Plan, ProjParams
    N, B, L, R = 512, 1, 5, 16
    gen = torch.Generator("cuda").manual_seed(7)
    V0 = torch.view_as_complex(torch.randn((1, N, N, 8, 2), device="cuda", generator=gen))
    y = torch.zeros((B, N, N), dtype=torch.complex64, device="cuda")
    prm = ProjParams(iters=2, lr=1e-2, eps=1e-1, w_kspace=0.0, w_image=0.0, tv_xy=1e-1, l1=1e-2, tv_eps=1e-2)
    out = []
    for Nf in (8, 688):
        plan = Plan(N, L, R, np.array([0.3]), np.linspace(-3, 3, Nf), np.zeros(B, dtype=np.int32), 1)
        V, _ = plan.proj_reconstruct(y, prm, V=V0.repeat(1, 1, 1, Nf // 8))
        plan.destroy()
        out.append(V)
    assert float((out[0] - V0).abs().max()) > 1e-3
    for f in range(0, 688, 8):
        assert float((out[1][..., f:f + 8] - out[0]).abs().max()) < 1e-6
