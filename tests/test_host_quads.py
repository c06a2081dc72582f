"""Host check of the interpolation's quads, their records and the producer's
ring schedule (tests/host/quads_check.cu, no GPU needed)."""
import os
import subprocess

import pytest

HOST = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host")


def test_quads_equal_a_direct_interpolation(tmp_path):
    from paper_2311_13177_gb300 import build as B
    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "quads_check")
    b = subprocess.run([nvcc, "-std=c++17", "-O1", "-x", "cu", "-I", B.CSRC, os.path.join(HOST, "quads_check.cu"),
                        os.path.join(HOST, "stubs.cu"), "-o", exe], capture_output=True, text=True, timeout=600)
    assert b.returncode == 0, b.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:]
