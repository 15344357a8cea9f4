"""The library's plans also run as replicas, one per GPU of a machine, where loads
that are multicast to a cluster's CTAs must not be used: no kernel has any."""
from __future__ import annotations

import os

PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_08471_gb300")


def test_no_multicast():
    files = [os.path.join(d, f) for d, _, fs in os.walk(PKG) for f in fs if f.endswith((".cu", ".cuh", ".h", ".py"))]
    assert len(files) > 10
    for path in files:
        with open(path) as f:
            assert "multicast" not in f.read(), path
