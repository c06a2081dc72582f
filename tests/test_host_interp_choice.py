"""Host check of the interpolation tiles and of the rule between tiles and quads
(tests/host/interp_choice_check.cu, no GPU needed)."""
import os
import subprocess

import pytest

HOST = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host")


def test_tiles_hold_every_sample_and_the_rule_follows_the_measurements(tmp_path):
    from paper_2311_13177_gb300 import build as B
    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "interp_choice_check")
    b = subprocess.run([nvcc, "-std=c++17", "-O1", "-x", "cu", "-I", B.CSRC, os.path.join(HOST, "interp_choice_check.cu"),
                        os.path.join(HOST, "stubs.cu"), "-o", exe], capture_output=True, text=True, timeout=600)
    assert b.returncode == 0, b.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.strip() == "OK", r.stdout[-3000:]
