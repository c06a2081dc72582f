"""The warp-specialised row kernel's walks of one, two, three, four and six voxels
(N = 16 to 192; the voxels in flight follow the length) against the per-row
kernel, whose arithmetic is the same: equal bit for bit, with and without time
neighbours, a dead lane and a ragged last run.  The loss sums a thread's terms in
FP32 over its walks, at most 60 of them here (one unit a CTA in the per-row
kernel, several in the other): 60 roundings of 6e-8 of positive terms, 5e-6."""
import numpy as np
import pytest
import torch

from helpers import random_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,Nf,T", [(16, 16, 3), (32, 15, 2), (48, 16, 3), (64, 32, 1), (64, 16, 3), (96, 16, 2),
                                    (128, 31, 3), (192, 16, 2)])
def test_both_row_kernels_give_the_same_volume(N, Nf, T):
    from paper_2311_13177_gb300 import Plan, ReconParams
    c = random_case(N, Nf, 6, 3, N, T, seed=N + Nf)
    q = ReconParams(iters=3, lr=1e-2, tv_xy=1e-2, tv_t=1e-2)
    y, got = torch.from_numpy(c["y"]).cuda(), []
    for kernel in (1, 2):
        plan = Plan(N, 3, N, c["theta"], c["delta"], c["blade_frame"], T, kb_width=8, row_kernel=kernel)
        got.append(plan.reconstruct(y, q))
        plan.destroy()
    assert torch.equal(got[0][0], got[1][0])
    assert np.max(np.abs(got[0][1] - got[1][1]) / np.abs(got[0][1])) < 5e-6
