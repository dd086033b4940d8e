"""The planes per CTA that the default configuration of a binary32 grid ranks:
one for every number of CTAs, so that a long grid is created as fast as a short one."""
import os
import subprocess

from paper_1709_09713_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_ranked_planes_per_cta(tmp_path):
    exe = str(tmp_path / "chunks_check")
    subprocess.run([build.nvcc(), "-O2", "-std=c++17", "--expt-relaxed-constexpr", *build.ARCH, "-I", build.CSRC, "-o", exe,
                    os.path.join(ROOT, "tests", "chunks_check.cu")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
