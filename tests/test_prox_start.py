"""The power prox starts from an FP32 root and corrects it with one full-precision power; how far off
the start may be (prox_reach in pdmcf_resident.cuh) has to leave less than half a last place. The
correction restated in 60 digits at that limit: both steps with FP64 iterates, one with FP32."""
import os
import re
from decimal import Decimal, getcontext

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_17996_gb300",
                   "csrc", "pdmcf_resident.cuh")


def _limits():
    text = open(SRC, encoding="utf-8").read()
    m = re.search(r"prox_reach\(\) \{ return sizeof\(P\) == 8 \? P\((\S+)\) : P\((\S+)\); \}", text)
    assert "fabs(d) * (c1 + P(1)) < prox_reach<P>()" in text
    return {64: Decimal(m.group(1)), 32: Decimal(m.group(2))}


def _root(y, c1):
    """t^(c1+1) (t + y) = 1 by Newton from the right, to 60 digits."""
    t = max(Decimal(0), -y) + 1
    for _ in range(400):
        p = t ** c1
        new = t - (p * t * (t + y) - 1) / (p * ((c1 + 2) * t + (c1 + 1) * y))
        if abs(new - t) < t * Decimal("1e-55"):
            return new
        t = new
    raise AssertionError("no root")


@pytest.mark.parametrize("bits", [64, 32])
@pytest.mark.parametrize("gamma", ["0.05", "0.1", "0.3", "0.7", "0.9", "0.95"])
def test_correction_at_the_limit(bits, gamma):
    getcontext().prec = 60
    g = Decimal(gamma)
    c1 = g / (1 - g)
    half_place = Decimal(2) ** (-53 if bits == 64 else -24)
    for y in map(Decimal, ("-5", "-1", "-0.1", "0", "0.1", "1", "5", "100")):
        t = _root(y, c1)
        a, b = c1 + 2, (c1 + 1) * y
        for side in (1, -1):
            t0 = t * (1 + side * _limits()[bits] / (c1 + 1))
            p0 = t0 ** c1
            t1 = t0 - (p0 * t0 * (t0 + y) - 1) / (p0 * (a * t0 + b))
            d = (t1 - t0) / t0
            p1 = p0 * (1 + c1 * d * (1 + (c1 - 1) * d / 2 * (1 + (c1 - 2) * d / 3)))
            z, p = t1, p1
            if bits == 64:
                z = t1 - (p1 * t1 * (t1 + y) - 1) / (p1 * (a * t1 + b))
                p = p1 * (1 + c1 * (z - t1) / t1)
            assert abs(z / t - 1) < half_place, (y, side)
            assert abs(t ** (c1 + 1) / (p * z) - 1) < half_place, (y, side)   # the traffic
