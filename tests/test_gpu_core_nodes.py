"""The FP32 form's cores on grids fine enough for 32-point blocks to be taken
through Chebyshev nodes, against the oracle: around the largest half-width that
is accepted (16 beta = 0.3: dnu = 3.6e-4 here), from few lines (block-edge gaps
between the rule's regions) to many, narrow to broad, ragged grid ends.  Bar:
the form's 1e-5 where the opacity exceeds 1e-8 of the maximum; the rule's own
share is 1.5e-7."""
import numpy as np
import pytest

import oracle
from paper_1503_03806_gb300 import synth
from tests.helpers import NTHREADS, Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dnu", [5e-5, 3.4e-4, 3.6e-4, 4e-4])
@pytest.mark.parametrize("n", [1, 40, 1500])
@pytest.mark.parametrize("P", [1e-6, 0.003, 0.1, 2.0])
def test_fine_grids(dnu, n, P):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1503_03806_gb300 import build
    build.build()
    from paper_1503_03806_gb300 import helk
    c = helk.Context(0)
    ng = 4000 + 13
    lines = synth.random_lines(n, 97, 5000.0, 5000.0 + ng * dnu)
    case = Case(1500.0, P, 18.0, (5000.0, dnu, ng), ("abs", 1.0))
    c.upload(lines)
    k = case.gpu(c, precision=helk.HELK_PREC_F32_KAHAN).cpu().numpy()
    c.close()
    ko, _, _ = oracle.opacity(lines, case.oracle_cond(), nthreads=NTHREADS)
    sel = ko > 1e-8 * ko.max()
    rel = np.abs(k[sel] / ko[sel] - 1.0)
    print("max %.2e rms %.2e" % (rel.max(), np.sqrt(np.mean(rel ** 2))))
    assert rel.max() < 1e-5


def test_batch_equals_singles_across_the_choice():
    # conditions on both sides of the kernel choice (Doppler widths ~ sqrt(T))
    from paper_1503_03806_gb300 import build
    build.build()
    from paper_1503_03806_gb300 import helk
    c = helk.Context(0)
    lines = synth.random_lines(300, 98, 5000.0, 5002.0)
    grid, T, P = (5000.0, 4e-4, 5000), [90.0, 900.0, 2500.0], [0.01, 0.1, 0.002]
    c.upload(lines)
    for order in ([0, 1, 2], [0, 0, 0], [2, 0, 1]):
        b = c.opacity_batch([T[k] for k in order], [P[k] for k in order], 18.0, ("abs", 1.0), grid,
                            precision=helk.HELK_PREC_F32_KAHAN).cpu().numpy().reshape(3, -1)
        for r, k in enumerate(order):
            one = c.opacity(T[k], P[k], 18.0, ("abs", 1.0), grid, precision=helk.HELK_PREC_F32_KAHAN).cpu().numpy()
            assert np.array_equal(b[r], one)
    c.close()
