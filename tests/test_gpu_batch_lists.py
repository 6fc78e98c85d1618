"""Batches on one context whose line list changes between calls: the buffers of a
captured sequence may have moved when a call of its shape comes back (a longer list
in between, or a single call), so each batch is compared, bit for bit, with a new
context's."""
import numpy as np
import pytest

from paper_1503_03806_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("cut", [("abs", 0.1), ("abs", 3.0)])
def test_lists_of_other_lengths_in_between(precision, cut):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1503_03806_gb300 import build
    build.build()
    from paper_1503_03806_gb300 import helk
    grid = (100.0, 0.01, 4000)
    T, P = np.linspace(300.0, 2000.0, 12), np.logspace(-3, 0.5, 12)
    lists = [synth.random_lines(n, 7 + i, 100.0, 140.0, with_elower=True, extra_fields=(i % 2 == 0))
             for i, n in enumerate((100, 5000, 100, 64, 5000, 40_000, 100, 5000))]
    out = torch.empty((12, grid[2]), dtype=torch.float64, device="cuda")
    c = helk.Context(0)
    for lines in lists:
        c.upload(lines)
        c.opacity(700.0, 0.2, 18.0, cut, grid, precision=precision)  # grows the buffers of one condition
        got = c.opacity_batch(T, P, 18.0, cut, grid, out=out, precision=precision).cpu().numpy()
        f = helk.Context(0)
        f.upload(lines)
        want = f.opacity_batch(T, P, 18.0, cut, grid, precision=precision).cpu().numpy()
        f.close()
        assert want.max() > 0 and np.array_equal(got, want), lines["nu0"].size
    c.close()
