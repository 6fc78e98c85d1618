"""Line fields past FP32's range in the FP32 form: lower-state energies up to
1e300, whose Boltzmann factor is 0 (or, at the reference temperature, 1), and
a line centre out there, leave the other lines' opacity as the FP64 form has it, at
the form's 1e-5, and no point without a number."""
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


@pytest.mark.parametrize("E", [1e30, 1e38, 3e38, 1e39, 1e200, 1e300])
@pytest.mark.parametrize("T", [40.0, 200.0, 296.0])
@pytest.mark.parametrize("cut", [("abs", 2.0), ("none",)])
def test_energies(ctx, E, T, cut):
    from paper_1503_03806_gb300 import helk
    lines = synth.random_lines(300, 3, 100.0, 130.0, with_elower=True)
    lines["E_lower"][::5] = E
    ctx.upload(lines)
    args = (T, 0.5, 18.0, cut, (100.0, 0.01, 3000))
    k64 = ctx.opacity(*args, q_ratio=0.7).cpu().numpy()
    k32 = ctx.opacity(*args, q_ratio=0.7, precision=helk.HELK_PREC_F32_KAHAN).cpu().numpy()
    sel = k64 > 1e-8 * k64.max()
    assert np.all(np.isfinite(k64)) and np.all(np.isfinite(k32)) and sel.sum() > 1000
    np.testing.assert_allclose(k32[sel], k64[sel], rtol=1e-5)


def test_centre(ctx):
    from paper_1503_03806_gb300 import helk
    lines = synth.random_lines(300, 3, 100.0, 130.0, with_elower=True)
    lines["nu0"][-1] = 1e39
    ctx.upload(lines)
    args = (700.0, 0.5, 18.0, ("abs", 2.0), (100.0, 0.01, 3000))
    k64 = ctx.opacity(*args).cpu().numpy()
    k32 = ctx.opacity(*args, precision=helk.HELK_PREC_F32_KAHAN).cpu().numpy()
    sel = k64 > 1e-8 * k64.max()
    assert np.all(np.isfinite(k32))
    np.testing.assert_allclose(k32[sel], k64[sel], rtol=1e-5)
