"""FP32 opacity of lists with masses per line on grids where lines reach the nodes of
the core kernel, where only the lightest do and where none do, the masses in any
order and changing from upload to upload, against the FP64 form at the FP32 form's
1e-5; a list of one mass against the call's mass."""
import numpy as np
import pytest

from paper_1503_03806_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dnu", [2e-4, 1e-3, 4e-3, 0.02, 0.2])
def test_masses(dnu):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1503_03806_gb300 import build
    build.build()
    from paper_1503_03806_gb300 import helk
    ctx = helk.Context(0)
    grid = (9000.0, dnu, 20_000)
    base = synth.random_lines(1500, 31, 9000.0, 9000.0 + 20_000 * dnu)
    rng = np.random.default_rng(7)
    for masses in ((300.0, 44.0), (300.0, 1.0), (18.0,), (44.0, 2.0), (300.0,)):
        lines = dict(base, mass=rng.choice(masses, 1500))
        ctx.upload(lines)
        args = (1800.0, 0.01, 18.0, ("abs", 400 * dnu), grid)
        k64 = ctx.opacity(*args).cpu().numpy()
        k32 = ctx.opacity(*args, precision=helk.HELK_PREC_F32_KAHAN).cpu().numpy()
        sel = k64 > 1e-8 * k64.max()
        np.testing.assert_allclose(k32[sel], k64[sel], rtol=1e-5)
        kb = ctx.opacity_batch([300.0, 1800.0], [0.1, 0.01], 18.0, args[3], grid, precision=helk.HELK_PREC_F32_KAHAN)
        assert np.array_equal(kb[1].cpu().numpy(), k32)
    ctx.close()
