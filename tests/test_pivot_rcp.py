"""Host check of the CholInv leaf's pivot arithmetic: 1/d in integers within
0.52 ulp over its range, 1/sqrt(d) and sqrt(d) within 0.55 ulp of the exact
values, and which pivots are left to divisions."""
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


def _bits(x):
    return struct.unpack("<q", struct.pack("<d", x))[0]


def _run(tmp_path, ds):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "pivot_rcp_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC,
                    os.path.join(HERE, "native", "pivot_rcp_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], input="".join(f"{_bits(d)}\n" for d in ds), capture_output=True, text=True,
                         check=True).stdout
    for d, ln in zip(ds, out.strip().split("\n")):
        w = ln.split()
        yield d, w[0] == "1", *(struct.unpack("<d", int(x, 16).to_bytes(8, "little"))[0] for x in w[1:])


def test_reciprocal_and_roots(tmp_path):
    rng = random.Random(11)
    ds = [math.ldexp(rng.uniform(1.0, 2.0), rng.randint(-998, 995)) for _ in range(20000)]
    ds += [math.ldexp(m, e) for e in (-999, -1, 0, 1, 2, 995)
           for m in (1.0, 1.0 + 2.0**-52, 2.0 - 2.0**-52, 1.5, 1.0 + 2.0**-23, 2.0 - 2.0**-23)]
    for d, ok, y, r, l in _run(tmp_path, ds):
        assert ok
        ulp = Fraction(math.ulp(y))
        assert abs(Fraction(y) - 1 / Fraction(d)) <= ulp * Fraction(52, 100), d
        # |r - 1/sqrt(d)| = |1/d - r^2| / (1/sqrt(d) + r) to first order
        assert abs(1 / Fraction(d) - Fraction(r) ** 2) <= 2 * Fraction(r) * Fraction(math.ulp(r)) * Fraction(55, 100), d
        assert abs(Fraction(d) - Fraction(l) ** 2) <= 2 * Fraction(l) * Fraction(math.ulp(l)) * Fraction(55, 100), d


def test_pivots_left_to_divisions(tmp_path):
    ds = [0.0, -0.0, -1.0, math.inf, -math.inf, math.nan, 5e-324, 2.0**-1000, 2.0**1000, -(2.0**-30)]
    assert [ok for _, ok, *_ in _run(tmp_path, ds)] == [False] * len(ds)
