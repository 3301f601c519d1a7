"""The whole-warp waits of the GEMM kernels, on barriers that do and do not complete (each wait ends by its own limit)."""
import os
import subprocess

import pytest

from paper_2505_19115_b200 import build

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_whole_warp_waits_end_alike_for_every_lane(tmp_path):
    exe = tmp_path / "bounded_waits_check"
    subprocess.check_call([build.NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O3", "-I", os.path.join(ROOT, "paper_2505_19115_b200", "csrc"),
                           os.path.join(ROOT, "tests", "native", "bounded_waits_check.cu"), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
