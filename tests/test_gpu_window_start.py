"""Windows that begin or end exactly on the grid's first or last point, and
windows of a single point (a zero cutoff on a grid point): the FP32 form covers
the points that the FP64 form covers, counts as many evaluations, and has its
values at the first point, for one call and for a batch."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("nu_min,dnu,n", [(0.0, 0.01, 300), (500.0, 0.01, 5000), (500.0, 1.0 / 128, 2000), (8.0, 0.5, 64)])
@pytest.mark.parametrize("c", [0, 1, 25, 100])
@pytest.mark.parametrize("kind", ["abs", "lorentz"])
def test_first_and_last_point(ctx, nu_min, dnu, n, c, kind):
    from paper_1503_03806_gb300 import helk
    grid = (nu_min, dnu, n)
    C = nu_min + c * dnu - nu_min  # the distance of grid point c from the first, as the arithmetic has it
    nu = np.array([nu_min + C, nu_min + (n - 1) * dnu - C, nu_min + 0.5 * n * dnu])
    nu = nu[nu > 0]
    lines = {"nu0": np.sort(nu), "S0": np.full(nu.size, 1e-20), "gamma_air": np.full(nu.size, 8.0 * dnu)}
    ctx.upload(lines)
    cut = ("abs", C) if kind == "abs" else ("lorentz", 1e9, C)
    P = 1.0
    k64 = ctx.opacity(296.0, P, 18.0, cut, grid).cpu().numpy()
    n64 = ctx.stats()[0]
    k32 = ctx.opacity(296.0, P, 18.0, cut, grid, precision=helk.HELK_PREC_F32_KAHAN).cpu().numpy()
    n32 = ctx.stats()[0]
    assert n64 == n32 and np.array_equal(k64 != 0, k32 != 0)
    if nu_min + C > 0:
        assert k64[0] > 0
    sel = k64 > 1e-8 * k64.max()
    np.testing.assert_allclose(k32[sel], k64[sel], rtol=1e-5)
    kb = ctx.opacity_batch([296.0, 296.0], [P, P], 18.0, cut, grid, precision=helk.HELK_PREC_F32_KAHAN).cpu().numpy()
    assert np.array_equal(kb[0], k32) and np.array_equal(kb[1], k32)


def test_zero_lorentz_cutoff(ctx):
    """P = 0 under the Lorentz cutoff: each line has the point it lies on."""
    from paper_1503_03806_gb300 import helk
    nu = 500.0 + np.array([0.0, 1.0, 3.0])
    ctx.upload({"nu0": nu, "S0": np.full(3, 1e-20), "gamma_air": np.full(3, 0.05)})
    grid, cut = (500.0, 0.25, 40), ("lorentz", 500.0, 100.0)
    k64 = ctx.opacity(296.0, 0.0, 18.0, cut, grid).cpu().numpy()
    k32 = ctx.opacity(296.0, 0.0, 18.0, cut, grid, precision=helk.HELK_PREC_F32_KAHAN).cpu().numpy()
    assert ctx.stats()[0] == 3
    assert np.array_equal(np.flatnonzero(k64), [0, 4, 12]) and np.array_equal(np.flatnonzero(k32), [0, 4, 12])
    np.testing.assert_allclose(k32[[0, 4, 12]], k64[[0, 4, 12]], rtol=1e-5)
