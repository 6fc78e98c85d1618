"""Line lists of several ordered runs (merged at upload, up to 16 runs) and of
more (radix-sorted): the same opacity, bit for bit, as the list sorted stably on
the host, with every optional field present and ties between and inside runs."""
import numpy as np
import pytest

from paper_1503_03806_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths", [[1, 1], [2, 1, 1], [5, 700, 3], [1000] * 4, [300] * 16, [300] * 17, [1] * 40])
@pytest.mark.parametrize("ties", [False, True])
def test_runs(lengths, ties):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1503_03806_gb300 import build
    build.build()
    from paper_1503_03806_gb300 import helk
    n = sum(lengths)
    rng = np.random.default_rng(n)
    lines = synth.random_lines(n, 3, 10.0, 60.0, with_elower=True, extra_fields=True)
    lines["mass"], lines["weight"] = rng.choice([2.0, 18.0], n), rng.uniform(0.1, 1.0, n)
    nu = rng.uniform(10.0, 60.0, n)
    if ties:
        nu = np.ceil(nu)
    at = 0
    for k in lengths:  # ordered runs, each starting below the end of the one before
        nu[at:at + k] = np.sort(nu[at:at + k])
        at += k
    if lengths == [1] * 40:
        nu = np.sort(nu)[::-1].copy()
    lines["nu0"] = nu
    order = np.argsort(nu, kind="stable")
    c = helk.Context(0)
    got = []
    for ls in (lines, {k: np.ascontiguousarray(v[order]) for k, v in lines.items()}):
        c.upload(ls)
        got.append(c.opacity(700.0, 0.5, 18.0, ("abs", 5.0), (10.0, 0.05, 1001)).cpu().numpy())
    c.close()
    assert got[0].max() > 0
    assert np.array_equal(got[0], got[1])
