"""The test for a physical state (rho > 0, p > 0) answers the same at every scale
of the state's units (compiled for the host; the kernels use the same source)."""
import os
import subprocess

from paper_1812_04789_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_physical_at_every_scale(tmp_path):
    exe = str(tmp_path / "physical_range")
    cmd = [build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
           os.path.join(HERE, "csrc", "physical_range.cu"), "-o", exe]
    subprocess.run(cmd, check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    print(r.stdout)
    assert r.returncode == 0, r.stdout + r.stderr
