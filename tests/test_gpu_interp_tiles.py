"""Plans that take interpolation tiles at the bin strides with quads (few samples
a frame, one line a blade, 64 bins): forward and gradient against the oracle at
both widths, odd counts, the wrapping last tile and ragged chunks, and a batch of
plans of both kinds against each plan's own run, bit for bit.

Tolerance: width 8's own error is 5e-8 and the transforms are at most 14 radix-2
stages of a few 6e-8 roundings, 2e-6 (width 6, error 6e-6 as the operator's
tests have it: 5e-5); the gradient adds the adjoint's: twice that."""
import numpy as np
import pytest
import torch

import oracle
from helpers import geometry, random_case, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,Nf,B,L,R,T,chunk,width", [
    (16, 8, 8, 1, 16, 8, 0, 8),
    (24, 15, 9, 3, 25, 9, 0, 8),      # a dead bin, odd counts, 2N = 48
    (32, 32, 8, 1, 33, 8, 0, 8),      # 12-row tiles: the last one wraps
    (32, 64, 8, 5, 29, 8, 0, 8),
    (16, 63, 16, 3, 16, 16, 0, 6),
    (48, 40, 6, 1, 48, 6, 32, 8),     # chunks of 32 and 8: the second at the run-time stride
    (32, 28, 8, 2, 32, 8, 16, 6),     # chunks of 16 and 12
])
def test_tiles_match_the_oracle(N, Nf, B, L, R, T, chunk, width):
    from paper_2311_13177_gb300 import Plan, ReconParams
    c = random_case(N, Nf, B, L, R, T, seed=N + Nf)
    c["theta"] = np.mod(np.arange(B) * 1.9416, np.pi)
    g = geometry(N, L, R, c["theta"], c["delta"], c["blade_frame"], T)
    plan = Plan(N, L, R, c["theta"], c["delta"], c["blade_frame"], T, bin_chunk=chunk, kb_width=width)
    V, y = (torch.from_numpy(c[k]).cuda() for k in ("V", "y"))
    p = dict(iters=1, tv_xy=1e-2, tv_t=1e-2)
    want, ref = oracle.recon.loss_and_grad(c["V"].astype(np.complex128), c["y"].astype(np.complex128), g,
                                           oracle.ReconParams(lr=1e-2, **p))
    got = plan.forward(V).cpu().numpy()
    loss, grad = plan.loss_grad(y, ReconParams(**p), V)
    plan.destroy()
    tol = 2e-6 if width == 8 else 5e-5
    assert rel(got, oracle.forward(c["V"].astype(np.complex128), g)) < tol
    assert abs(loss - want) < 2 * tol * abs(want)
    assert rel(grad.cpu().numpy(), ref) < 2 * tol


@pytest.mark.parametrize("Nf,width", [(64, 8), (32, 6), (8, 8)])
def test_a_batch_of_tiles_and_quads_equals_each_plan_alone(Nf, width):
    from paper_2311_13177_gb300 import Plan, ReconParams, prop_reconstruct_batch
    plans, ys, q = [], [], ReconParams(iters=4, lr=1e-2, tv_xy=1e-3, tv_t=1e-3)
    for B, L, T in ((8, 1, 8), (24, 8, 1), (16, 3, 16), (48, 4, 1)):  # tiles, quads, tiles, quads
        c = random_case(32, Nf, B, L, 32, T, seed=B + L)
        plans.append(Plan(32, L, 32, c["theta"], c["delta"], c["blade_frame"], T, kb_width=width))
        ys.append(torch.from_numpy(c["y"]).cuda())
    together, _ = prop_reconstruct_batch(plans, ys, [q] * len(plans), trace=False)
    for p, y, V in zip(plans, ys, together):
        assert torch.equal(p.reconstruct(y, q)[0], V)
        p.destroy()
