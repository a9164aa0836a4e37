"""The limb sums of 128-bit integers and the fast conversion to double against exact integers (CPU only)."""
import os
import shutil
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
M64 = (1 << 64) - 1


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    out = tmp_path_factory.mktemp("wide") / "wide_harness"
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2003_00082_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "wide_sum_harness.cpp"), "-o", str(out)])
    return str(out)


def run(harness, groups):
    text = ""
    for E, xs in groups:
        text += f"E {E}\n" + "".join(f"X {x & M64:x} {(x >> 64) & M64:x}\n" for x in xs) + "S\n"
    out = subprocess.run([harness], input=text, capture_output=True, text=True, check=True).stdout.split()
    return [tuple(int(h, 16) for h in out[i:i + 4]) for i in range(0, len(out), 4)]


def nearest(x, E):
    """bits of the double nearest to x 2^(E - 1129)"""
    e = E - 1129
    v = Fraction(x) * (Fraction(2) ** e)
    try:
        f = v.numerator / v.denominator      # int / int rounds correctly
    except OverflowError:
        f = float("inf") if v > 0 else float("-inf")
    return struct.unpack("<Q", struct.pack("<d", f))[0]


@pytest.mark.parametrize("E", [1, 54, 107, 108, 500, 1023, 1900, 2040, 2046])
def test_limb_sums_and_conversion(harness, E):
    rng = np.random.default_rng(E)
    groups = [(E, [0]), (E, [1]), (E, [-1]), (E, [-1] * 32), (E, [(1 << 122) - 1] * 32), (E, [-(1 << 122)] * 32)]
    for lead in range(1, 127):      # every position of the leading bit, ties and near ties among them
        top = 1 << lead
        for x in (top, top - 1, top + (top >> 53), top + (top >> 53) + 1, top + (top >> 53) - 1, top + 3 * (top >> 53)):
            groups.append((E, [x]))
            groups.append((E, [-x]))
    for _ in range(300):
        k = int(rng.integers(1, 33))
        width = int(rng.integers(1, 122))
        xs = [int.from_bytes(rng.bytes(16), "little", signed=True) >> (127 - width) for _ in range(k)]
        groups.append((E, xs))
    for (_, xs), (lo, hi, fast, general) in zip(groups, run(harness, groups)):
        total = sum(xs)
        assert (lo, hi) == (total & M64, (total >> 64) & M64)
        ref = nearest(total, E)
        assert fast == general
        if total == 0 or (ref >> 52) & 0x7FF:      # a normal number (the general conversion rounds a subnormal one twice)
            assert fast == ref, (E, hex(total))
