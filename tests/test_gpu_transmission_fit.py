"""Transmission from the fit over numbers of points, masses and bins on both sides
of its two rules (threads that share a mass, blocks with or without coefficients),
against FP64 sums at the bar of the fit's own test."""
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


@pytest.mark.parametrize("ng", [1, 2, 15, 16, 17, 64, 65, 200, 1000])
@pytest.mark.parametrize("nm", [1, 4, 30, 64, 65, 300])
@pytest.mark.parametrize("nbins", [1, 300])
def test_rules(ctx, ng, nm, nbins):
    import torch
    c = np.tile(np.array([[-46.0, 4.0, 0.5], [-45.0, 0.01, 0.0], [-44.0, -6.0, 1.0]]), (nbins // 3 + 1, 1))[:nbins]
    m = np.concatenate([[0.0], np.logspace(14, 26, nm)])[:nm]
    _, fit = ctx.transmission(nbins, m, coeffs=torch.from_numpy(c).cuda(), ng=ng)
    t = 2.0 * (np.arange(ng) + 0.5) / ng - 1.0
    got = fit.cpu().numpy()
    for b in range(min(nbins, 3)):
        k = np.exp(c[b, 0] + c[b, 1] * t + c[b, 2] * (2.0 * t * t - 1.0))
        want = np.exp(-k[None, :] * m[:, None]).mean(axis=1)
        pos = want > 1e-290
        rel = np.abs(got[b][pos] / want[pos] - 1.0)
        assert np.all(rel <= 1e-12 + 2e-14 * np.abs(np.log(want[pos]))), rel.max()
        assert np.array_equal(got[b::3], np.broadcast_to(got[b], got[b::3].shape))
