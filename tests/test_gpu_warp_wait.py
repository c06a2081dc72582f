"""The give-up path of the warps that wait for staged items: one decision a warp
(tests/device/warp_wait_check.cu; every wait in it is bounded)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_a_warp_gives_up_as_a_whole(tmp_path):
    from paper_2311_13177_gb300 import build as B
    exe = str(tmp_path / "warp_wait_check")
    b = subprocess.run([B.nvcc(), *B.ARCH, "-std=c++17", "-O2", "-I", B.CSRC,
                        os.path.join(HERE, "device", "warp_wait_check.cu"), "-o", exe],
                       capture_output=True, text=True, timeout=600)
    assert b.returncode == 0, b.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "OK", r.stdout[-2000:] + r.stderr[-2000:]
