"""FP64 opacity where the device has room for the point-by-point route's buffers but
not for those of the interpolated wings: the call (and a batch) still runs, as it did
before there were wings, with the point-by-point kernels; with room again it takes the
wings."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_no_room_for_the_wings():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1503_03806_gb300 import build
    build.build()
    from paper_1503_03806_gb300 import helk
    n = 3_000_000  # 96 MB of wing records a condition
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    u = lambda a, b: torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (b - a) + a
    lines = {"nu0": torch.sort(u(0.05, 30_000.0)).values, "S0": 10.0 ** u(-26, -19), "gamma_air": u(0.02, 0.1)}
    grid, cut = (10_000.0, 0.01, 50_000), ("abs", 1.0)
    ctx = helk.Context(0)
    ctx.upload(lines)
    T, P = [900.0, 1500.0], [0.3, 1.0]
    out, outs = torch.empty(grid[2], dtype=torch.float64, device="cuda"), torch.empty((2, grid[2]), dtype=torch.float64,
                                                                                     device="cuda")
    # buffers and kernels of the point-by-point route (windows of 10 points a side)
    ctx.opacity(T[0], P[0], 18.0, ("abs", 0.1), grid, out=out)
    ctx.opacity_batch(T, P, 18.0, ("abs", 0.1), grid, out=outs)
    ctx.sync()
    torch.cuda.synchronize()
    hog = []
    while torch.cuda.mem_get_info()[0] > 48 << 20:
        try:
            hog.append(torch.empty(torch.cuda.mem_get_info()[0] - (32 << 20), dtype=torch.uint8, device="cuda"))
        except RuntimeError:
            break
    free = torch.cuda.mem_get_info()[0]
    one = ctx.opacity(T[0], P[0], 18.0, cut, grid, out=out).cpu().numpy()
    both = ctx.opacity_batch(T, P, 18.0, cut, grid, out=outs).cpu().numpy()
    ctx.sync()
    del hog
    torch.cuda.empty_cache()
    assert free < 90 << 20
    assert np.array_equal(one, both[0])
    wings = ctx.opacity_batch(T, P, 18.0, cut, grid, out=outs).cpu().numpy()
    assert np.array_equal(ctx.opacity(T[0], P[0], 18.0, cut, grid, out=out).cpu().numpy(), wings[0])
    assert one.min() > 0 and not np.array_equal(both, wings)
    np.testing.assert_allclose(both, wings, rtol=1e-9)
    ctx.close()
