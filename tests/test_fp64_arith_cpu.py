"""The FP64 form's arctangent and sine series restated on the CPU (table and coefficients read from the
source; fused multiply-adds through the extended type) against the exact functions."""
import os
import re

import numpy as np
import pytest

SRC = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_08500_gb300", "csrc",
                        "rr_device.cuh")).read()
L = np.longdouble

pytestmark = pytest.mark.skipif(np.finfo(L).nmant < 63, reason="needs an extended type")


def fma(a, b, c):
    return np.float64(L(a) * L(b) + L(c))


def table():
    body = re.search(r"kAtanTab\[33\] = \{(.*?)\}", SRC, re.S).group(1)
    return [float(x) for x in body.replace("\n", " ").split(",") if x.strip()]


def atan2_upper64(y, x, tab):
    ax = abs(x)
    steep, left = y > ax, x < 0
    mx, mn = (y, ax) if steep else (ax, y)
    j = int(np.clip(np.rint(np.float32(32) * np.float32(mn) / np.float32(mx)), 0, 32))
    t0 = j / 32
    u = np.float64(fma(-t0, mx, mn) / fma(t0, mn, mx))
    v = u * u
    p = fma(v * v, fma(v, 1 / 9, -1 / 7), fma(v, 1 / 5, -1 / 3))
    c0 = np.pi / 2 if steep else (np.pi if left else 0.0)
    c1 = 6.123233995736766e-17 if steep else (1.2246467991473532e-16 if left else 0.0)
    th = -tab[j] if steep != left else tab[j]
    s = c0 + th
    e = (c0 - s) + th + c1
    a = fma(u * v, p, u)
    return s + ((-a if steep != left else a) + e)


def test_atan_table():
    t = table()
    assert len(t) == 33
    ref = np.arctan(np.arange(33, dtype=L) / 32)
    assert all(float(r) == v for r, v in zip(ref, t))


def test_atan2_upper64_within_two_ulp():
    tab = table()
    rng = np.random.default_rng(1)
    worst = 0.0
    for _ in range(20000):
        y, x = abs(rng.normal()) * 10 ** rng.uniform(-9, 1), rng.normal() * 10 ** rng.uniform(-9, 1)
        ref = np.arctan2(L(y), L(x))
        worst = max(worst, float(abs(L(atan2_upper64(y, x, tab)) - ref) / L(np.spacing(float(ref)))))
    assert worst < 2.0
    assert atan2_upper64(0.0, 1.0, tab) == 0.0 and atan2_upper64(1.0, 0.0, tab) == np.pi / 2
    assert atan2_upper64(0.0, -1.0, tab) == np.pi


def test_sine_series_is_exact_to_rounding_on_the_unit_interval():
    """Every denominator of the two series is the factorial it stands for, and the truncated sums hold."""
    body = SRC[SRC.index("void half_angle_SV64("):]
    body = body[:body.index("sincos(")]
    den = [int(float(d)) for _, d in re.findall(r"(-?)1\.0 / ([0-9]+)\.0", body)]
    import math
    fact = {math.factorial(n): n for n in range(2, 21)}
    assert sorted(fact[d] for d in den) == sorted(list(range(3, 20, 2)) + list(range(4, 21, 2)))
    sign = {fact[int(float(d))]: (-1.0 if s else 1.0) for s, d in re.findall(r"(-?)1\.0 / ([0-9]+)\.0", body)}
    x = np.linspace(-1, 1, 4001, dtype=L)
    S = x + sum(L(sign[n]) * x ** n / L(math.factorial(n)) for n in range(3, 20, 2))
    V = x * x / 2 + sum(L(sign[n]) * x ** n / L(math.factorial(n)) for n in range(4, 21, 2))
    assert np.abs(S - np.sin(x)).max() < 5e-19
    assert np.abs(V - 2 * np.sin(x / 2) ** 2).max() < 5e-19
