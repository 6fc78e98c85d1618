"""The two forms of the FP32 core kernel (voigt_core.cuh), in FP64 against the
exact w(z): the series in powers of e^x inside core_inner(y), the 8-node
Gauss-Hermite rule outside, and the polynomials of its exponential and sine
(coefficients read from the source)."""
import os
import re

import numpy as np
import pytest
from numpy.polynomial import polynomial as P
from numpy.polynomial.hermite import hermgauss

special = pytest.importorskip("scipy.special")
SRC = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1503_03806_gb300", "csrc",
                        "voigt_core.cuh")).read()


def inner_bound(y):
    return np.where(y >= 4.5, 0.0, np.where(y >= 1.0, 23.5, 29.5 + 0.8 * np.maximum(0.0, -np.log(np.maximum(y, 1e-8)
                                                                                                * 100.0))))


def samples():
    rng = np.random.default_rng(916)
    y = np.concatenate([10.0 ** rng.uniform(-9, 1, 40000), [1e-30, 1e-12, 0.999, 1.0, 4.499, 4.5]])
    x = rng.uniform(0.0, 10.0, y.size)
    ok = x * x + y * y < 100.0
    return x[ok], y[ok]


def test_inner_series():
    x, y = samples()
    m = x * x < inner_bound(y)
    x, y = x[m], y[m]
    n = np.arange(1, 23)[:, None]
    k = 1.0 / np.pi  # 2 h / pi
    S1 = sum(np.exp(-(0.5 * i) ** 2) / ((0.5 * i) ** 2 + y * y) for i in range(1, 14))
    A = special.erfcx(y) - k * y * S1
    D = k / y - 2.0 * A
    c = 0.5 * k * y * np.exp(-n * n / 4.0) / (n * n / 4.0 + y * y)
    s = np.sin(x * y)
    pos = (c * np.exp(n * x)).sum(0)
    neg = (c[:8] * np.exp(-n[:8] * x)).sum(0)
    K = np.exp(-x * x) * (A + D * s * s + pos + neg)
    ref = special.wofz(x + 1j * y).real
    assert np.max(np.abs(K / ref - 1.0)) < 2e-8


def test_outer_rule():
    x, y = samples()
    m = x * x >= inner_bound(y)
    x, y = x[m], y[m]
    t, w = hermgauss(8)
    K = (y / np.pi * (w / ((x[:, None] - t) ** 2 + (y * y)[:, None])).sum(1))
    K = K + np.where(y < 1e-8, np.exp(-x * x), 0.0)
    ref = special.wofz(x + 1j * y).real
    assert np.max(np.abs(K / ref - 1.0)) < 4e-8


def _floats(text):
    return [float(v.rstrip("f")) for v in re.findall(r"-?\d+\.\d+(?:e-?\d+)?f", text)]


def test_exponential_and_sine_polynomials():
    body = SRC[SRC.index("core_exp(float z"):SRC.index("core_pow2")]
    q = [v for v in _floats(body) if abs(v) in (0.5,) or 1e-3 < abs(v) < 0.2]
    q = [v for v in q if v not in (1.0,)]
    coef = sorted(q, reverse=True)  # 1/2, 1/6, 1/24, ..
    assert len(coef) == 5
    r = np.linspace(-0.34658, 0.34658, 5001)
    p = r + r * r * P.polyval(r, coef)
    assert np.max(np.abs(p - np.expm1(r)) / np.exp(r)) < 1.2e-8
    body = SRC[SRC.index("float s = fmaf("):SRC.index("return core_gauss(x, x2) * (")]
    c = _floats(body)  # highest first
    assert len(c) == 4
    t = np.linspace(1e-3, np.pi / 2, 5001)
    s = t + t * t * t * P.polyval(t * t, c[::-1])
    assert np.max(np.abs(s / np.sin(t) - 1.0)) < 1.2e-8
