"""Bins too large for shared memory, split by value: sizes at the edges of the
number of parts, spectra whose keys crowd (zeros, runs of one value, a narrow
range that one bucket of the split holds), and sorting in place.  Sorted values
bit for bit, tables at the bounds of the k-table tests."""
import numpy as np
import pytest

from paper_1503_03806_gb300 import synth
from tests.test_gpu_kdist import check_kdist

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


@pytest.mark.parametrize("nb", [22_400, 30_001, 57_344, 57_345])
def test_sizes(ctx, nb):
    check_kdist(ctx, synth.uniform_kappa(2 * nb, nb), 2, 20)


@pytest.mark.parametrize("kind", ["zeros", "mostly_zeros", "constant", "runs", "narrow", "outlier"])
def test_crowded_keys(ctx, kind):
    nb = 30_000
    k = synth.uniform_kappa(2 * nb, 7).reshape(2, nb)
    rng = np.random.default_rng(3)
    if kind == "zeros":
        k[:, rng.random(nb) < 0.3] = 0.0
    elif kind == "mostly_zeros":
        k[:, rng.random(nb) < 0.97] = 0.0
    elif kind == "constant":
        k[0] = 3.0e-21
    elif kind == "runs":
        k[:, :12_000] = k[:, :1]
    elif kind == "narrow":  # one value apart from the rest: a single bucket of the split
        k = 1.0e-20 * (1.0 + 1.0e-9 * rng.random((2, nb)))
        k[:, 0] = 1.0e-40
    else:
        k[:, 5] = 1.0e-200
    check_kdist(ctx, np.ascontiguousarray(k.reshape(-1)), 2, 12, floor=1e-60)


def test_sorted_output_onto_the_input(ctx):
    import ctypes
    import torch
    from paper_1503_03806_gb300 import helk
    k = torch.from_numpy(synth.uniform_kappa(2 * 30_000, 9)).cuda()
    want = torch.sort(k.view(2, -1), dim=1).values
    coef = torch.empty((2, 12), dtype=torch.float64, device="cuda")
    p = ctypes.c_void_p(k.data_ptr())
    assert helk.helk_kdist(ctx.h, p, 60_000, 2, 12, 1e-250, ctypes.c_void_p(coef.data_ptr()), None, 0, p) == helk.HELK_OK
    ctx.sync()
    assert torch.equal(k.view(2, -1), want)
