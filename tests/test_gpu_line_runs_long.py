"""Lists on both sides of the length from which more than 8 ordered runs are sorted
rather than merged, and of the lengths at which fewer fields are reordered a launch:
the same opacity, bit for bit, as the list sorted on the host; and 16 runs of a long
list take no longer to upload than 17 (with a margin for noise)."""
import numpy as np
import pytest

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


def runs_of(n, runs, seed):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    u = lambda a, b: torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (b - a) + a
    nu = u(0.05, 3000.0)
    if runs:
        nu = torch.cat([torch.sort(v).values for v in nu.chunk(runs)])
    return {"nu0": nu, "S0": 10.0 ** u(-26, -19), "gamma_air": u(0.02, 0.1), "E_lower": u(0.0, 1e4),
            "mass": torch.where(u(0, 1) < 0.5, 18.0, 44.0), "weight": u(0.1, 1.0)}


@pytest.mark.parametrize("n", [2 ** 18, 2 ** 18 + 1, 2_800_000, 2_800_001, 4_200_000, 8_400_000])
@pytest.mark.parametrize("runs", [8, 9, 16, 0])
def test_order(ctx, n, runs):
    import torch
    lines = runs_of(n, runs, 3)
    order = torch.argsort(lines["nu0"], stable=True)
    got = []
    for ls in (lines, {k: v[order].contiguous() for k, v in lines.items()}):
        ctx.upload(ls)
        got.append(ctx.opacity(700.0, 0.5, 18.0, ("abs", 0.02), (0.0, 0.05, 60000)).clone())
    assert got[0].max().item() > 0 and torch.equal(got[0], got[1])


def test_cost(ctx):
    import time
    best = []
    for runs in (16, 17):
        lines = runs_of(4_000_000, runs, 5)
        ts = []
        for _ in range(5):
            t0 = time.perf_counter()
            ctx.upload(lines)
            ts.append(time.perf_counter() - t0)
        best.append(min(ts))
    assert best[0] < 1.25 * best[1], best
