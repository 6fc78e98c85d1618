"""More column masses than one launch has blocks for (more than 65535 blocks of 8
warps of 32 masses): every one of them, for a sorted bin and for one that takes the
plain sum, and from a fit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_many_column_masses():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1503_03806_gb300 import build
    build.build()
    from paper_1503_03806_gb300 import helk
    nm = 65535 * 8 * 32 + 33 * 257
    m = np.linspace(0.0, 30.0, nm)
    k = np.array([[0.5, 1.0, 1.0, 2.0], [2.0, 0.25, 1.0, 3.0]])  # sorted, unsorted
    ctx = helk.Context(0)
    direct, fit = ctx.transmission(2, m, sorted_k=torch.from_numpy(k.reshape(-1)).cuda(),
                                   coeffs=torch.tensor([[0.0], [-1.0]], dtype=torch.float64, device="cuda"), ng=2)
    for b in range(2):
        want = np.zeros(nm)
        for v in k[b]:
            want += 0.25 * np.exp(-v * m)
        np.testing.assert_allclose(direct[b].cpu().numpy(), want, rtol=1e-12)
        np.testing.assert_allclose(fit[b].cpu().numpy(), np.exp(-np.exp(-float(b)) * m), rtol=1e-12)
    ctx.close()
