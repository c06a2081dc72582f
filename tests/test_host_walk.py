"""Host check of the updates' walks along x1 (tests/host/walk_check.cu, no GPU
needed)."""
import os
import subprocess

import pytest

HOST = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host")


def test_walks_cover_a_row_once(tmp_path):
    from paper_2311_13177_gb300 import build as B
    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "walk_check")
    b = subprocess.run([nvcc, "-std=c++17", "-O1", "-x", "cu", "-I", B.CSRC, os.path.join(HOST, "walk_check.cu"), "-o",
                        exe], capture_output=True, text=True, timeout=600)
    assert b.returncode == 0, b.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.strip() == "OK", r.stdout[-3000:]
