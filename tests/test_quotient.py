"""Host check of the least-squares solve's quotients: from the divisor's reciprocal
and one correction, bit for bit the division, for divisors in 2^-500 .. 2^500 and
quotients in the normal range."""
from __future__ import annotations

import math
import os
import random
import shutil
import struct
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1710_08471_gb300", "csrc")


def _bits(x):
    return struct.unpack("<q", struct.pack("<d", x))[0]


def test_quotients_are_correctly_rounded(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "quotient_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC,
                    os.path.join(HERE, "native", "quotient_check.cpp"), "-o", exe], check=True)
    rng = random.Random(5)
    edge = [1.0, 1.0 + 2.0**-52, 2.0 - 2.0**-52, 1.5, 1.0 + 2.0**-23, 2.0 - 2.0**-23, 4.0 / 3.0, 3.0]
    pairs = [(a, d) for a in edge for d in edge] + [(0.0, d) for d in edge]
    pairs += [(math.ldexp(rng.uniform(1, 2), rng.randint(-490, 490)) * rng.choice([-1, 1]),
               math.ldexp(rng.uniform(1, 2), rng.randint(-490, 490))) for _ in range(100000)]
    out = subprocess.run([exe], input="".join(f"{_bits(a)} {_bits(d)}\n" for a, d in pairs), capture_output=True,
                         text=True, check=True).stdout.split("\n")
    for (a, d), ln in zip(pairs, out):
        q, t = ln.split()
        assert q == t, (a, d)
