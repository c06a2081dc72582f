"""The spread whose items the CTAs claim at run time (plans with many items a
CTA): the counter has to be back at zero after every launch, or later adjoints
would skip items without an error.  The two full-size benchmark plans have too
few items to claim; the plan here has two thirds more than a GB300 needs, which
the list builder is asked on the host (no GPU), so that the test cannot lose its
subject unnoticed.

Tolerance: width 8's own error is 5e-8 and the transforms are 20 radix-2 stages
of a few 6e-8 roundings: 2e-6."""
import os
import subprocess

import numpy as np
import pytest
import torch

import oracle
from helpers import geometry, rel

HOST = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host")
N, NF, B, L, R, W = 384, 64, 32, 32, 384, 8


def _items(tmp_path, sms):
    from paper_2311_13177_gb300 import build as BLD
    try:
        nvcc = BLD.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "spread_claim_count")
    b = subprocess.run([nvcc, "-std=c++17", "-O1", "-x", "cu", "-I", BLD.CSRC, os.path.join(HOST, "spread_claim_count.cu"),
                        os.path.join(HOST, "stubs.cu"), "-o", exe], capture_output=True, text=True, timeout=600)
    assert b.returncode == 0, b.stderr[-3000:]
    r = subprocess.run([exe, *map(str, (N, NF, B, L, R, W, sms))], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout
    return map(int, r.stdout.split())


def test_the_plan_claims_its_items_with_a_margin(tmp_path):
    items, least = _items(tmp_path, 152)
    assert items > 1.5 * least


@pytest.mark.gpu
def test_repeated_adjoints_of_claimed_items(tmp_path):
    from paper_2311_13177_gb300 import Plan
    items, least = _items(tmp_path, torch.cuda.get_device_properties(0).multi_processor_count)
    assert items > 1.25 * least
    theta, delta = np.pi * np.arange(B) / B, np.linspace(-4.0, 4.0, NF)
    rng = np.random.default_rng(3)
    y = (rng.standard_normal((B, L, R)) + 1j * rng.standard_normal((B, L, R))).astype(np.complex64)
    plan = Plan(N, L, R, theta, delta, kb_width=W)
    yd = torch.from_numpy(y).cuda()
    first = plan.adjoint(yd)
    for _ in range(3):
        assert torch.equal(plan.adjoint(yd), first)
    plan.destroy()
    v = first.cpu().numpy().reshape(-1)
    q = rng.choice(v.size, 128, replace=False)
    assert rel(v[q], oracle.adjoint_at(y.astype(np.complex128), geometry(N, L, R, theta, delta), q)) < 2e-6
