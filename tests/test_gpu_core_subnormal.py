"""FP32 form without pressure: the far end of a core, where e^{-x^2} falls from the
smallest normal FP32 number (x^2 = 87) to e^-100 = 3.7e-44, is small but not zero:
where the FP32 form is zero the FP64 form is below the smallest subnormal number,
1.4e-45 of the line's strength.  On a fine grid (sums at nodes) and a coarse one,
with the route by windows of 40 points too."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dnu", [1e-4, 1e-3])
@pytest.mark.parametrize("cut", [("none",), ("abs", 0.04)])
@pytest.mark.parametrize("count", [False, True])
def test_far_end_of_an_undamped_core(dnu, cut, count):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1503_03806_gb300 import build
    build.build()
    from paper_1503_03806_gb300 import helk
    ctx = helk.Context(0)
    n = int(0.3 / dnu)
    ctx.upload({"nu0": np.array([1000.05, 1000.15]), "S0": np.array([1e-20, 1e-20]), "gamma_air": np.array([0.07, 0.07])})
    args = (1500.0, 0.0, 18.0, cut, (1000.0, dnu, n))
    k64 = ctx.opacity(*args).cpu().numpy()
    k32 = ctx.opacity(*args, precision=helk.HELK_PREC_F32_KAHAN, count_regions=count).cpu().numpy()
    top = k64.max()  # about the scale: 2^E is at most twice it
    assert np.all(k64[k32 == 0.0] < 2.0 * 1.5e-45 * top)
    assert ((k64 > 0) & (k64 < 1.2e-38 * top) & (k64 > 1e-43 * top)).sum() > 10 or cut[0] == "abs"
    ctx.close()
