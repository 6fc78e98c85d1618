"""FP64 opacity of lists with few lines to a tile, on both sides of the rule that
leaves them to the point-by-point kernels: values against the counting call (always
point by point) at 1e-9; lists of one length whose lines lie elsewhere, so that a
batch of one shape takes one route and then the other, against a new context, bit for
bit; and the cost of a sparse list, which is at most that of the counting call and a
margin."""
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


@pytest.mark.parametrize("n,counts", [(300, (1, 15, 19, 20, 21, 40)), (30_000, (1, 50, 75, 85, 100, 400)),
                                      (300_000, (1, 100, 260, 280, 1000))])
@pytest.mark.parametrize("half", [24.0, 2500.0])
def test_values(ctx, n, counts, half):
    for nl in counts:
        ctx.upload(synth.random_lines(nl, 5, 3000.0, 3000.0 + n * 0.01))
        args = (900.0, 0.4, 18.0, ("abs", half * 0.01), (3000.0, 0.01, n))
        ref = ctx.opacity(*args, count_regions=True).cpu().numpy()
        k = ctx.opacity(*args).cpu().numpy()
        assert np.array_equal(k != 0, ref != 0), nl
        np.testing.assert_allclose(k, ref, rtol=1e-9)
        kb = ctx.opacity_batch([900.0, 500.0], [0.4, 0.4], 18.0, args[3], args[4]).cpu().numpy()
        assert np.array_equal(kb[0], k), nl


def test_routes_in_turn(ctx):
    from paper_1503_03806_gb300 import helk
    grid, cut = (3000.0, 0.01, 20_000), ("abs", 1.0)
    near, far = synth.random_lines(2000, 5, 3000.0, 3200.0), synth.random_lines(2000, 6, 6000.0, 9000.0)
    far["nu0"][:3] = [3010.0, 3100.0, 3150.0]
    far["nu0"].sort()
    for lines in (near, far, near, far):
        ctx.upload(lines)
        got = ctx.opacity_batch([900.0, 500.0], [0.4, 0.1], 18.0, cut, grid).cpu().numpy()
        one = ctx.opacity(900.0, 0.4, 18.0, cut, grid).cpu().numpy()
        f = helk.Context(0)
        f.upload(lines)
        want = f.opacity_batch([900.0, 500.0], [0.4, 0.1], 18.0, cut, grid).cpu().numpy()
        f.close()
        assert want.max() > 0 and np.array_equal(got, want) and np.array_equal(got[0], one)


@pytest.mark.parametrize("n,nl", [(3_000_000, 1), (3_000_000, 100), (300_000, 10)])
def test_cost(ctx, n, nl):
    import torch
    ctx.upload(synth.random_lines(nl, 5, 1.0, n * 0.01))
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    best = []
    for count in (False, True):
        ms = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ctx.opacity(1500.0, 1.0, 18.0, ("abs", 25.0), (0.0, 0.01, n), out=out, count_regions=count)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        best.append(min(ms))
    assert best[0] < 1.5 * best[1], best
