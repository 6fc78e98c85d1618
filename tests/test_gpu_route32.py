"""FP32 opacity on both sides of the rule that chooses between interpolated wings and
the point-by-point kernels: numbers of lines around its thresholds on grids of its
three kinds, and a band of a long list, against the FP64 counting call at the form's
1e-5; one call and a batch bit for bit."""
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


def check(ctx, lines, half, grid):
    from paper_1503_03806_gb300 import helk
    f32 = helk.HELK_PREC_F32_KAHAN
    ctx.upload(lines)
    cut = ("abs", half * grid[1])
    ref = ctx.opacity(1100.0, 0.3, 18.0, cut, grid, count_regions=True).cpu().numpy()
    k = ctx.opacity(1100.0, 0.3, 18.0, cut, grid, precision=f32).cpu().numpy()
    sel = ref > 1e-8 * ref.max()
    np.testing.assert_allclose(k[sel], ref[sel], rtol=1e-5)
    kb = ctx.opacity_batch([1100.0, 400.0], [0.3, 0.1], 18.0, cut, grid, precision=f32).cpu().numpy()
    assert np.array_equal(kb[0], k)


@pytest.mark.parametrize("n,half,counts", [(2500, 64.0, (90, 99, 100, 120, 400)), (40_000, 300.0, (500, 1450, 1550, 3000)),
                                           (200_000, 3000.0, (2000, 4900, 5100, 20_000)),
                                           (400_000, 2000.0, (2000, 7700, 8200, 30_000))])
def test_values(ctx, n, half, counts):
    for nl in counts:
        check(ctx, synth.random_lines(nl, 5, 3000.0, 3000.0 + n * 0.01), half, (3000.0, 0.01, n))


@pytest.mark.parametrize("nl", [1000, 30_000, 200_000])
def test_band(ctx, nl):
    check(ctx, synth.random_lines(nl, 5, 0.0, 30_000.0), 1500.0, (10_000.0, 0.01, 90_001))
