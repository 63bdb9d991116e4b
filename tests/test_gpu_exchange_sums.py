"""The persistent smoother's sums over the CTAs are FP64 sums of what the CTAs
publish, also for FP32 vectors (bars beside the program)."""
import os
import subprocess

import pytest

from paper_1812_04789_gb300 import build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_sums_over_ctas_are_fp64(tmp_path):
    exe = str(tmp_path / "exchange_sums")
    cmd = [build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
           "-I", build.INCLUDE, os.path.join(HERE, "csrc", "exchange_sums.cu"), "-o", exe]
    subprocess.run(cmd, check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    print(r.stdout)
    assert r.returncode == 0, r.stdout + r.stderr
