"""Transmission by blocks of neighbouring values: bins at the edges of a block
(64 values), with gaps that make a block wide, ties and few masses, against
FP64 sums; the fit at point counts around its blocks and its shared memory."""
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


@pytest.mark.parametrize("nb", [1, 2, 63, 64, 65, 129, 2049])
@pytest.mark.parametrize("nm", [1, 7, 300])
def test_direct_block_edges(ctx, nb, nm):
    import torch
    rng = np.random.default_rng(nb)
    bins = [np.sort(10.0 ** rng.uniform(-28, -18, nb)), np.sort(rng.uniform(1e-20, 1.001e-20, nb)),
            np.sort(np.where(rng.random(nb) < 0.5, 1e-24, 10.0 ** rng.uniform(-20, -19.99, nb)))]
    k = np.stack(bins)
    m = np.concatenate([[0.0], np.logspace(15, 27, nm)])[:nm]
    direct, _ = ctx.transmission(len(bins), m, sorted_k=torch.from_numpy(k.reshape(-1)).cuda())
    want = np.exp(-k[:, None, :].astype(np.longdouble) * m[None, :, None]).mean(axis=2).astype(np.float64)
    np.testing.assert_allclose(direct.cpu().numpy(), want, rtol=1e-12, atol=1e-300)


@pytest.mark.parametrize("ng", [1, 15, 16, 17, 1000, 9500, 14000])
def test_fit_blocks(ctx, ng):
    import torch
    c = np.array([[-46.0, 4.0, 0.5], [-45.0, 0.01, 0.0], [-44.0, -6.0, 1.0]])
    m = np.concatenate([[0.0], np.logspace(14, 26, 200)])
    _, fit = ctx.transmission(3, m, coeffs=torch.from_numpy(c).cuda(), ng=ng)
    t = 2.0 * (np.arange(ng) + 0.5) / ng - 1.0
    k = np.exp(c[:, :1] + c[:, 1:2] * t + c[:, 2:] * (2.0 * t * t - 1.0))
    want = np.stack([np.exp(-k[b][None, :] * m[:, None]).mean(axis=1) for b in range(3)])
    got = fit.cpu().numpy()
    pos = want > 1e-290
    rel = np.abs(got[pos] / want[pos] - 1.0)
    assert np.all(rel <= 1e-12 + 2e-14 * np.abs(np.log(want[pos]))), rel.max()
