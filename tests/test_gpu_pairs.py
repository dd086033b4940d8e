"""The double-float split of a binary64 value used by the stages: hi + lo is
the value to 48 bits, or to 2^-126, over the binary32 range, and zeros, overflow, infinities
and NaNs keep their meaning."""
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_split_of_binary64_values(tmp_path):
    from paper_1709_09713_gb300 import build

    exe = str(tmp_path / "split_check")
    subprocess.run([build.nvcc(), "-O3", "-std=c++17", *build.ARCH, "-I", build.CSRC, "-o", exe,
                    os.path.join(ROOT, "tests", "split_check.cu")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
