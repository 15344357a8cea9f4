"""Host check of the Q-form's conversion with one shift per group of outputs:
(X 2^24 + Y) 2^E with the low bits of Y rounded off at the shift the group's
largest |X| allows, then one correct rounding, against exact rational
arithmetic; zeros, cancellation, the largest accumulators (16384 columns),
subnormal and overflowing results."""
from __future__ import annotations

import math
import os
import random
import shutil
import struct
import subprocess
from fractions import Fraction

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1710_08471_gb300", "csrc")
MAX_CHUNK_X = sum((g + 1) * 2**21 * 256 ** (3 - g) for g in range(4))  # groups 0-3 of one chunk of 128
MAX_CHUNK_Y = sum((g + 1) * 2**21 * 256 ** (6 - g) for g in range(4, 7))


def _nearest(x):
    try:
        return float(x)  # Fraction to the nearest double, subnormals included
    except OverflowError:
        return math.inf if x > 0 else -math.inf


def test_group_conversion(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "group_shift_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC,
                    os.path.join(HERE, "native", "group_shift_check.cpp"), "-o", exe], check=True)
    rng = random.Random(7)
    cases = []
    for chunks in (1, 2, 3, 8, 128):
        mx, my = MAX_CHUNK_X * chunks, MAX_CHUNK_Y * chunks
        for E in (-62, -120, 0, 500, -1000, -1090, -1130, 960, 1000):
            vals = [(0, 0, 0), (0, 0, mx), (mx, my, mx), (-mx, -my, mx), (mx, -my, 0), (1, 0, 0), (0, 1, 0), (0, -1, mx),
                    (-1, my, mx), (1, -my, 0), (1, 0, mx)]
            for _ in range(150):
                x, y = rng.randint(-mx, mx) >> rng.randint(0, 47), rng.randint(-my, my) >> rng.randint(0, 40)
                vals.append((x, y, rng.choice([0, x, mx, rng.randint(-mx, mx) >> rng.randint(0, 30)])))
            cases += [(X, Y, H, E) for X, Y, H in vals]
    out = subprocess.run([exe], input="".join("%d %d %d %d\n" % c for c in cases), capture_output=True, text=True,
                         check=True).stdout.strip().split("\n")
    for (X, Y, H, E), ln in zip(cases, out):
        s, bits = ln.split()
        sh = 24 - int(s)
        got = struct.unpack("<d", int(bits, 16).to_bytes(8, "little"))[0]
        exact = Fraction(X * 2**24 + Y) * Fraction(2) ** E
        Z = (X << (24 - sh)) + ((Y + ((1 << sh) >> 1)) >> sh)
        assert 0 <= sh <= 24 and abs(Z) < 2**63
        # as small a shift as 62 bits allow, or none
        assert sh == 0 or max(abs(X), abs(H)) >= 2 ** (61 - (24 - sh)) - 1
        rounded = Fraction(Z) * Fraction(2) ** (E + sh)
        if Z == 0:
            assert got == 0.0 and abs(exact) <= Fraction(2) ** (E + sh - 1)
            continue
        assert abs(rounded - exact) <= Fraction(2) ** (E + sh) / 2
        z = abs(float(Z))  # as the hardware rounds it; out of the normal range the exact conversion takes over
        e = math.frexp(z)[1] + E + sh
        assert got == (_nearest(rounded) if -1021 <= e <= 1024 else _nearest(exact))
