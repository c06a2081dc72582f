"""Grids of which the samples reach only a part (Plan::grid_used): the column
passes and the spread skip the blocks of 16 rows x 2 columns that no
footprint meets.  Forward and adjoint against the oracle for every bin stride
with grouped lists and every kind of column pass, with a grid left full of
NaN by the call before.

Tolerance: width 8's own error is 5e-8; the transforms are at most
2 log2(1024) = 20 radix-2 stages of a few 6e-8 roundings each, so 2e-6."""
import numpy as np
import pytest
import torch

import oracle
from helpers import geometry, random_case, rel

pytestmark = pytest.mark.gpu
TOL = 2e-6


@pytest.mark.parametrize("N,Nf,B,L,R,T,chunk", [
    (16, 8, 1, 1, 16, 1, 0),      # 2N = 32: two blocks a column
    (24, 7, 2, 3, 25, 2, 0),      # 2N = 48, bin stride 8, odd counts
    (48, 16, 3, 4, 48, 3, 0),     # 2N = 96, one blade a frame
    (64, 64, 2, 5, 64, 1, 0),     # bin stride 64: eight column tiles share a pair of columns
    (96, 31, 2, 3, 97, 1, 0),     # 2N = 192, bin stride 32 with a dead bin
    (64, 20, 2, 4, 64, 2, 16),    # chunks 16 + 4 share the blocks
    (192, 8, 2, 3, 60, 2, 0),     # 2N = 384: 24 values a thread
    (256, 8, 1, 3, 80, 1, 0),     # 2N = 512: 32 values a thread
    (384, 8, 1, 2, 64, 1, 0),     # 2N = 768: adjoint columns without staged input
    (512, 8, 1, 2, 64, 1, 0),     # 2N = 1024: 64 blocks a column
    (32, 6, 2, 3, 32, 2, 0),      # bin stride 6: the whole grid
])
def test_forward_and_adjoint_on_a_partly_used_grid(N, Nf, B, L, R, T, chunk):
    from paper_2311_13177_gb300 import Plan
    c = random_case(N, Nf, B, L, R, T, seed=N + Nf)
    c["theta"] = c["theta"] + 0.4   # no blade along an axis
    g = geometry(N, L, R, c["theta"], c["delta"], c["blade_frame"], T)
    plan = Plan(N, L, R, c["theta"], c["delta"], c["blade_frame"], T, bin_chunk=chunk, kb_width=8)
    V, y = (torch.from_numpy(c[k]).cuda() for k in ("V", "y"))
    bad = torch.full_like(V, float("nan"))
    assert torch.isnan(plan.forward(bad).real).all()
    got_V = plan.adjoint(y).cpu().numpy()
    plan.forward(bad)
    got_y = plan.forward(V).cpu().numpy()
    plan.destroy()
    assert rel(got_y, oracle.forward(c["V"].astype(np.complex128), g)) < TOL
    assert rel(got_V, oracle.adjoint(c["y"].astype(np.complex128), g)) < TOL
