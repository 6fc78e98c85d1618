"""The FP32 form's line preparation (pairs of FP32, windows by a product with
1 / dnu) against the FP64 form's: the same window for every line, so the same
points are non-zero, also where a bound falls on a grid point or next to one;
strengths over the whole FP64 range, energies whose exponential leaves it,
masses, weights and exponents per line.  Values: each FP32 record entry is
rounded once from <= 1e-9 (2^-24 = 6e-8), and the profile itself keeps the
form's 1e-5 where the opacity exceeds 1e-8 of the largest.
"""
import numpy as np
import pytest

from paper_1503_03806_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1503_03806_gb300 import build
    build.build()
    from paper_1503_03806_gb300 import helk
    c = helk.Context(0)
    yield c
    c.close()


def both(ctx, lines, T, P, cut, grid, q=1.0, mass=18.0):
    from paper_1503_03806_gb300 import helk
    ctx.upload(lines)
    k64 = ctx.opacity(T, P, mass, cut, grid, q_ratio=q).cpu().numpy()
    k32 = ctx.opacity(T, P, mass, cut, grid, q_ratio=q, precision=helk.HELK_PREC_F32_KAHAN).cpu().numpy()
    return k64, k32


@pytest.mark.parametrize("dnu", [0.01, 1.0 / 128, 0.003, 0.7])
@pytest.mark.parametrize("nu_min", [0.0, 1234.567])
def test_windows(ctx, dnu, nu_min):
    n = 2000
    for c, w in ((1000, 100), (3, 150), (1998, 90), (-50, 120), (2050, 100), (700, 64), (1000, 5000)):
        for eps in (0.0, 1e-16, -1e-16, 1e-13, -1e-13, 0.5 * dnu):
            nu = nu_min + c * dnu
            if not nu > 0.0:
                continue
            lines = {"nu0": np.array([nu * (1 + eps) if abs(eps) < 1e-3 else nu + eps]), "S0": np.array([1e-20]),
                     "gamma_air": np.array([8.0 * dnu])}
            k64, k32 = both(ctx, lines, 296.0, 1.0, ("abs", w * dnu), (nu_min, dnu, n))
            assert np.array_equal(k64 != 0, k32 != 0), (c, w, eps)


@pytest.mark.parametrize("cut", [("abs", 5.0), ("lorentz", 300.0, 20.0), ("none",)])
@pytest.mark.parametrize("T,E_max", [(200.0, 1e7), (1700.0, 2e4)])
def test_fields(ctx, cut, T, E_max):
    n = 900
    rng = np.random.default_rng(5)
    lines = synth.random_lines(n, 41, 100.0, 160.0, with_elower=True, extra_fields=True)
    lines["mass"] = rng.choice([2.0, 18.0, 44.0], n)
    lines["weight"] = 10.0 ** rng.uniform(-6, 0, n)
    lines["weight"][::50] = 0.0
    lines["E_lower"] = rng.choice([0.0, 1.5, 900.0, 2e4, E_max], n)
    lines["S0"] = 10.0 ** rng.uniform(-30, -18, n)
    lines["S0"][::7] = 10.0 ** rng.uniform(-320, -300, len(lines["S0"][::7]))
    for scale in (1.0, 1e-270, 1e250):
        scaled = dict(lines, S0=lines["S0"] * scale)
        k64, k32 = both(ctx, scaled, T, 0.7, cut, (100.0, 0.01, 6001), q=0.37)
        sel = k64 > 1e-8 * k64.max()
        assert sel.sum() > 1000
        np.testing.assert_allclose(k32[sel], k64[sel], rtol=1e-5)
