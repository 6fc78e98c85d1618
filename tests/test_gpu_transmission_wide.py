"""Transmission of bins that span so many decades that most differences from the
smallest value are below 2^-100 of the largest (FP64 terms): any number of them,
few and many masses, against extended-precision sums; and their cost, which is at
most that of the plain FP64 sum of as many values (an unsorted bin) and a factor
for noise."""
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


@pytest.mark.parametrize("tiny", [1, 31, 32, 33, 1000])
@pytest.mark.parametrize("nm", [1, 5, 40, 300])
def test_values(ctx, tiny, nm):
    import torch
    rng = np.random.default_rng(tiny)
    bins = [np.concatenate([np.full(7, 1e-70), np.sort(10.0 ** rng.uniform(-69.5, -52, tiny)),
                            np.sort(10.0 ** rng.uniform(-24, -18, 90))]),
            np.sort(10.0 ** rng.uniform(-78, -18, tiny + 97))]
    k = np.stack(bins)
    m = np.concatenate([[0.0], np.logspace(15, 72, nm)])[:nm]
    direct, _ = ctx.transmission(2, m, sorted_k=torch.from_numpy(k.reshape(-1)).cuda())
    want = np.exp(-k[:, None, :].astype(np.longdouble) * m[None, :, None]).mean(axis=2).astype(np.float64)
    np.testing.assert_allclose(direct.cpu().numpy(), want, rtol=1e-12, atol=1e-300)


@pytest.mark.parametrize("nbins,nb,nm", [(1, 100_000, 1), (1, 100_000, 30), (300, 10_000, 4), (300, 10_000, 300)])
def test_cost(ctx, nbins, nb, nm):
    import torch
    rng = np.random.default_rng(1)
    wide = np.sort(10.0 ** rng.uniform(-78, -18, (nbins, nb)), axis=1)
    plain = wide[:, ::-1].copy()
    m = np.logspace(14, 30, nm)
    best = []
    for k in (wide, plain):
        t = torch.from_numpy(k.reshape(-1)).cuda()
        ms = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ctx.transmission(nbins, m, sorted_k=t)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        best.append(min(ms))
    assert best[0] < 2.0 * best[1], best
