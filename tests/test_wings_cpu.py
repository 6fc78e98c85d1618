"""The interpolation behind the wings route, in FP64: the truncation bounds
its kernels rely on (panels at least eta half-widths from the poles, P
Chebyshev nodes), for a Lorentzian with its poles in any direction, and the
exactness of the parent-to-child step."""
import os
import re

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1503_03806_gb300", "csrc")


def basis(P, x):
    t = np.cos((2 * np.arange(P) + 1) * np.pi / (2 * P))
    w = (-1.0) ** np.arange(P) * np.sin((2 * np.arange(P) + 1) * np.pi / (2 * P))
    d = x[:, None] - t[None, :]
    d[d == 0] = 1e-300
    L = w / d
    return t, L / L.sum(1, keepdims=True)


@pytest.mark.parametrize("P,eta,bound", [(12, 3.0, 2.4e-8), (16, 5.0, 6e-15)])
def test_truncation_bound(P, eta, bound):
    x = np.linspace(-1.0, 1.0, 801)
    t, L = basis(P, x)
    worst = 0.0
    for th in np.linspace(0.0, np.pi / 2, 31):
        for r in (eta, 1.5 * eta, 4.0 * eta):
            f = lambda v: 1.0 / ((v - r * np.cos(th)) ** 2 + (r * np.sin(th)) ** 2)
            worst = max(worst, np.max(np.abs(L @ f(t) / f(x) - 1.0)))
    assert worst < bound, worst


def test_nodes_in_the_source():
    src = open(os.path.join(CSRC, "k_wings.cu")).read()
    vals = re.search(r"W32_T\[W32_P\] = \{(.*?)\}", src, re.S).group(1)
    got = np.array([float(v.strip().rstrip("f")) for v in vals.split(",")])
    assert np.max(np.abs(got - np.cos((2 * np.arange(12) + 1) * np.pi / 24))) < 1e-8


def test_child_step_is_exact_for_the_interpolant():
    P = 12
    t, _ = basis(P, np.zeros(1) + 0.3)
    rng = np.random.default_rng(0)
    v = rng.uniform(1.0, 2.0, P)
    x = np.linspace(-0.99, 0.99, 64)
    for side in (-0.5, 0.5):
        _, M = basis(P, side + 0.5 * t)
        _, Lc = basis(P, x)
        _, Lp = basis(P, side + 0.5 * x)
        assert np.max(np.abs(Lc @ (M @ v) - Lp @ v)) < 1e-11
