"""K-Planes render and parameter gradients against the oracle at the sizes
where the kernels' tiles and their choice can go wrong: bins kept in registers
(8, 16; runs of 8 or 16) and not, strips and frame batches with remainders,
more frames than are staged at once, feature counts from 1 to 32.

Tolerance: products of six FP32 factors (6 roundings of 6e-8) in sums of at
most 1e4 terms of random sign, whose rounding errors add up like a random walk
(1e2 times 6e-8 against a sum that grows the same way): below 1e-6; 1e-5 asked."""
import numpy as np
import pytest
import torch

from helpers import kplanes_pack, random_case, rel
from oracle import kplanes as kp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,Nf,T,F,S", [
    (24, 8, 5, 3, 2),     # Q = 6, a strip and a frame batch with remainders
    (16, 16, 18, 16, 2),  # Q = 32: 16 of the 18 frames staged at once, one column a thread in the render
    (16, 32, 6, 1, 1),    # Q = 1, two runs of 16 bins, general W kernel
    (24, 40, 3, 8, 1),    # five runs of 8 bins
    (32, 16, 4, 8, 2),    # the usual features
    (16, 1, 1, 2, 1),     # one bin, one frame
    (16, 13, 2, 8, 2),    # general kernels
    (16, 64, 2, 16, 2),   # largest bin and feature counts
    (96, 8, 3, 4, 1),     # X kernel: image rows in three equal runs
    (256, 8, 6, 1, 1),    # and in runs of 86, 86 and 84
])
def test_render_and_gradients(N, Nf, T, F, S):
    from paper_2311_13177_gb300 import Plan
    c = random_case(N, Nf, 2, 2, 8, T, seed=N + Nf)
    plan = Plan(N, 2, 8, c["theta"], c["delta"], c["blade_frame"], T)
    rng = np.random.default_rng(Nf + T)
    prm = kp.init_params(N, Nf, T, rng, F=F, scales=S, spread=0.3)
    gV = (rng.standard_normal((T, N, N, Nf)) + 1j * rng.standard_normal((T, N, N, Nf))).astype(np.complex64)
    flat = torch.from_numpy(kplanes_pack(prm).astype(np.complex64)).cuda()
    V = plan.kplanes_render(flat, F, S).cpu().numpy()
    G = plan.kplanes_vjp(flat, torch.from_numpy(gV).cuda(), F, S).cpu().numpy()
    again = plan.kplanes_vjp(flat, torch.from_numpy(gV).cuda(), F, S).cpu().numpy()
    plan.destroy()
    assert rel(V, kp.render(prm, N, Nf, T)) < 1e-5
    assert rel(G, kplanes_pack(kp.vjp(prm, gV.astype(np.complex128), N, Nf, T))) < 1e-5
    assert np.array_equal(G, again)
