"""Both sides of the rule by which transmission makes the coefficients of a bin's
blocks -- few and many masses, short and long bins, few and many bins, and the two
kernels that make them -- against extended-precision sums; few masses launch two
kernels, as they did without blocks."""
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


@pytest.mark.parametrize("nbins", [1, 13, 200])
@pytest.mark.parametrize("nb", [1, 65, 2048, 2049, 4100])
@pytest.mark.parametrize("nm", [1, 11, 12, 13])
def test_values(ctx, nbins, nb, nm):
    import torch
    rng = np.random.default_rng(nb + nm)
    k = np.sort(10.0 ** rng.uniform(-28, -18, (nbins, nb)), axis=1)
    k[0, : nb // 2] = k[0, 0]
    m = np.concatenate([[0.0], np.logspace(16, 25, nm)])[1 - nm:] if nm > 1 else np.array([1e20])
    before = ctx.launch_count()
    direct, _ = ctx.transmission(nbins, m, sorted_k=torch.from_numpy(k.reshape(-1)).cuda())
    if nm < 12 and nb <= 2048:
        assert ctx.launch_count() - before == 2
    got = direct.cpu().numpy()
    for b in sorted({0, nbins // 2, nbins - 1}):
        want = np.exp(-k[b][None, :].astype(np.longdouble) * m[:, None]).mean(axis=1).astype(np.float64)
        np.testing.assert_allclose(got[b], want, rtol=1e-12, atol=1e-300)
