"""The integer stencil sums of csrc/stencil_int.cuh against exact rational
arithmetic (host build), and the GPU build bit for bit against the host's."""
import math
import os
import struct
import subprocess
from fractions import Fraction

import pytest

from paper_1709_09713_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("stencil") / "stencil_check")
    subprocess.run([build.nvcc(), "-O2", "-std=c++17", "--expt-relaxed-constexpr", *build.ARCH, "-I", build.CSRC, "-o",
                    out, os.path.join(ROOT, "tests", "stencil_check.cu")], check=True)
    return out


# units of 2^-56 of the largest exponent 2^E that the cut values may lose: the sum of the weights
LOST = (18, 64, 34, 18)


def test_sums_against_exact_arithmetic(exe):
    text = subprocess.run([exe], capture_output=True, text=True, check=True, timeout=120).stdout
    checked = 0
    for line in text.splitlines():
        x = [struct.unpack("<d", struct.pack("<Q", int(w, 16)))[0] for w in line.split()]
        v, r = x[:5], x[5:]
        if not all(map(math.isfinite, v)):
            used = [k for k in range(5) if not math.isfinite(v[k])]
            assert math.isfinite(r[0]) == (used == [2]) and not math.isfinite(r[1])
            continue
        if max(map(abs, v)) > 1e300:  # the plain sums, which may overflow
            continue
        m2, m1, c, p1, p2 = map(Fraction, v)
        first = 8 * (p1 - m1) - (p2 - m2)
        want = (first, 16 * (p1 + m1) - (p2 + m2) - 30 * c, (p2 + m2) - 16 * (p1 + m1), first)
        for k in range(4):
            near = v if k == 1 else v[:2] + v[3:]
            top = max(math.frexp(a)[1] - 1 if a else -1100 for a in near)
            unit = Fraction(2) ** (max(top, 66 - 1023) - 56)
            off = abs(Fraction(r[k]) - want[k])
            spread = top - min(math.frexp(a)[1] - 1 if a else top for a in near)
            lost = 0 if spread <= 4 and top > -900 else LOST[k] * unit
            # half a unit in the last place of the result, and what was cut
            assert off <= abs(want[k]) / 2**53 * (1 + Fraction(1, 2**50)) + lost * (1 + Fraction(1, 2**52)), (v, k, r[k])
        checked += 1
    assert checked > 25000


def test_sums_of_eight_values(exe):
    """The binary64 x2 helper sums: weights 18 on each of two values a neighbour."""
    text = subprocess.run([exe, "eight"], capture_output=True, text=True, check=True, timeout=120).stdout
    checked = 0
    for line in text.splitlines():
        x = [struct.unpack("<d", struct.pack("<Q", int(w, 16)))[0] for w in line.split()]
        v, r = x[:8], x[8]
        if not all(map(math.isfinite, v)) or max(map(abs, v)) > 1e300:  # the plain sums
            continue
        m2, m1, p1, p2 = (Fraction(v[k]) + Fraction(v[4 + k]) for k in range(4))
        want = 8 * (p1 - m1) - (p2 - m2)
        tops = [math.frexp(a)[1] - 1 if a else -1100 for a in v]
        unit = Fraction(2) ** (max(max(tops), 66 - 1023) - 56)
        spread = max(tops) - min(t for t, a in zip(tops, v) if a) if any(v) else 0
        lost = 0 if spread <= 4 and max(tops) > -900 else 36 * unit
        assert abs(Fraction(r) - want) <= abs(want) / 2**53 * (1 + Fraction(1, 2**50)) + lost * (1 + Fraction(1, 2**52)), (v, r)
        checked += 1
    assert checked > 25000


@pytest.mark.gpu
def test_gpu_equals_host(exe):
    r = subprocess.run([exe, "gpu"], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
