"""Transmission of bins that take the plain FP64 sum (unsorted, or with a negative
value): lengths around the four-at-a-time loop, numbers of masses that no power of
two shares out; and the cost at 300 masses, which is ten times that at 30."""
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


@pytest.mark.parametrize("nb", [1, 2, 31, 33, 127, 128, 129, 257, 1000])
@pytest.mark.parametrize("nbins,nm", [(1, 1), (2, 37), (301, 300), (301, 333)])
def test_values(ctx, nb, nbins, nm):
    import torch
    rng = np.random.default_rng(nb)
    k = 10.0 ** rng.uniform(-24, -18, (nbins, nb))
    k[:, 0] = -1e-22  # (a bin of one value is sorted)
    k[1::3] = np.sort(np.abs(k[1::3]), axis=1)  # every third bin by blocks
    m = np.concatenate([[0.0], np.logspace(14, 22, nm)])[:nm]
    direct, _ = ctx.transmission(nbins, m, sorted_k=torch.from_numpy(k.reshape(-1)).cuda())
    got = direct.cpu().numpy()
    for b in list(range(min(nbins, 4))) + [nbins - 1]:
        want = np.exp(-k[b][None, :].astype(np.longdouble) * m[:, None]).mean(axis=1).astype(np.float64)
        np.testing.assert_allclose(got[b], want, rtol=1e-12)
    assert np.all(np.isfinite(got)) and np.allclose(got[:, 0], 1.0, rtol=1e-13)


def test_cost_is_proportional(ctx):
    import torch
    rng = np.random.default_rng(1)
    t = torch.from_numpy(10.0 ** rng.uniform(-28, -18, 300 * 10_000)).cuda()
    best = []
    for nm in (30, 300):
        m = np.logspace(14, 30, nm)
        ms = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ctx.transmission(300, m, sorted_k=t)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        best.append(min(ms))
    assert best[1] < 1.2 * 10 * best[0], best
