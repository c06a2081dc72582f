"""Host check of the grid blocks that the column passes and the spread are
limited to (tests/host/used_blocks_check.cu, no GPU needed)."""
import os
import subprocess

import pytest

HOST = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host")


def test_used_blocks_hold_every_footprint_and_the_lists_fill_them(tmp_path):
    from paper_2311_13177_gb300 import build as B
    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "used_blocks_check")
    b = subprocess.run([nvcc, "-std=c++17", "-O1", "-x", "cu", "-I", B.CSRC, os.path.join(HOST, "used_blocks_check.cu"),
                        os.path.join(HOST, "stubs.cu"), "-o", exe], capture_output=True, text=True, timeout=600)
    assert b.returncode == 0, b.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:]
