"""Sources of kernels that may be set up while their predecessor still writes
their inputs (launch_chained): nothing in them, comments aside, asks for the
read-only load path, whose data must not change during the kernel's lifetime."""
from __future__ import annotations

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_08471_gb300", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        s = f.read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", s, flags=re.S))


def _with_includes(name, seen):
    """The file and the project headers that it includes."""
    if name in seen:
        return
    seen[name] = _code(name)
    for inc in re.findall(r'#include "([^"/]+)"', seen[name]):
        if os.path.exists(os.path.join(CSRC, inc)):
            _with_includes(inc, seen)


def test_no_read_only_loads_in_chained_kernels():
    chained = [f for f in sorted(os.listdir(CSRC)) if f.endswith(".cu") and "grid_chain()" in _code(f)]
    assert len(chained) >= 6  # Gram, Q-form, GEMM, CholInv and its leaf, least-squares tail
    seen = {}
    for f in chained:
        _with_includes(f, seen)
    bad = {f: w for f, s in seen.items() for w in ("__ldg", "__restrict__", "ld.global.nc") if w in s}
    assert not bad, bad
