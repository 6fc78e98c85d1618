"""Both sides of the rule that chooses between interpolated wings and
point-by-point sums: half-widths around 24 points (FP64 form) and 64 points, and
around 43 lines to a point (FP32 form), against the counting call, which always
evaluates point by point in FP64.  FP64: 1e-9, the form's bar against the oracle;
FP32: its 1e-5 where the opacity exceeds 1e-8 of the maximum."""
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


@pytest.mark.parametrize("half", [22, 23.99, 24.01, 33, 63.99, 64.01, 100])
@pytest.mark.parametrize("n,nlines", [(3001, 600), (100_003, 20_000), (100_003, 60_000)])
def test_both_sides(ctx, half, n, nlines):
    from paper_1503_03806_gb300 import helk
    dnu = 0.01
    ctx.upload(synth.random_lines(nlines, 12, 3000.0, 3000.0 + n * dnu))
    args = (1200.0, 0.3, 18.0, ("abs", half * dnu), (3000.0, dnu, n))
    ref = ctx.opacity(*args, count_regions=True).cpu().numpy()
    k64 = ctx.opacity(*args).cpu().numpy()
    k32 = ctx.opacity(*args, precision=helk.HELK_PREC_F32_KAHAN).cpu().numpy()
    assert np.array_equal(k64 != 0, ref != 0)
    sel = ref > 0
    np.testing.assert_allclose(k64[sel], ref[sel], rtol=1e-9)
    sel = ref > 1e-8 * ref.max()
    np.testing.assert_allclose(k32[sel], ref[sel], rtol=1e-5)
