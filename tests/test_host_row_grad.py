"""Host check of the rule between the fused gradient row kernel and the separate
passes (tests/host/row_grad_check.cu, no GPU needed)."""
import os
import subprocess

import pytest

HOST = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host")


def test_the_rule_follows_the_measurements(tmp_path):
    from paper_2311_13177_gb300 import build as B
    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    B.build()
    obj = os.path.join(B.OBJDIR, "fft.o")
    if not os.path.exists(obj):
        B.build(force=True)
    exe = str(tmp_path / "row_grad_check")
    cmd = [nvcc, *B.ARCH, "-std=c++17", "-O1", "-cudart", "shared", "-I", B.CSRC, "-I", os.path.join(B.HERE, "..", "include"),
           os.path.join(HOST, "fake_runtime.cpp"), os.path.join(HOST, "row_grad_check.cu"), obj, "-o", exe]
    b = subprocess.run(cmd, capture_output=True, text=True, timeout=900)
    assert b.returncode == 0, b.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "OK", r.stdout[-3000:] + r.stderr[-2000:]
