"""The rule by which the FP32 form's core sums take a line on a 32-point block
through 10 Chebyshev nodes: the interpolation error relative to the profile,
for every block the rule accepts.  The remainder of the Gaussian part is
(2 x h)^10 / (10! 2^9) of it (h the block's half-width, 2 x h <= 1.5: 3.1e-8);
where the block lies farther out the Gaussian is at most e^-7 sqrt(pi) x^2 of
the profile, so the bound is 1.5e-7 at every point."""
import numpy as np
import pytest
from scipy.special import wofz


@pytest.mark.parametrize("y", [1e-9, 1e-6, 1e-4, 1e-3, 0.01, 0.05, 0.3, 1.0, 3.0, 9.0])
def test_rule(y):
    P = 10
    k = 2 * np.arange(P) + 1
    t, w = np.cos(k * np.pi / (2 * P)), (-1.0) ** np.arange(P) * np.sin(k * np.pi / (2 * P))
    p = (np.arange(32) - 15.5) / 16.0
    d = w / (p[:, None] - t[None, :])
    L = d / d.sum(1, keepdims=True)
    taken = 0
    for h in (0.3, 0.25, 0.1, 0.03):
        for c in np.arange(0.0, 9.0, 0.11):
            x = c + h * p
            xmax, xmin = np.abs(x).max(), (0.0 if x[0] * x[-1] <= 0 else np.abs(x).min())
            if not (2 * xmax * h <= 1.5 or xmin * xmin >= 7 - np.log(y)):
                continue
            taken += 1
            K = wofz(x + 1j * y).real
            err = np.abs(L @ wofz(c + h * t + 1j * y).real / K - 1)
            assert err.max() < 1.5e-7, (h, c, err.max())
    assert taken > 20
