"""Lists of a few hundred thousand lines in 9 or more ordered runs, on both sides of the
number of runs up to which such a length is merged: the same opacity, bit for bit, as the
list sorted on the host; and 9 runs of 4e5 lines take less time to upload than 17, which
are sorted (0.71 of it measured)."""
import pytest

from test_gpu_line_runs_long import ctx, runs_of  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,runs", [(375_000, 16), (375_001, 16), (400_000, 15), (400_000, 16),
                                    (1_000_000, 11), (1_000_000, 12), (3_000_000, 9), (3_000_001, 9)])
def test_order(ctx, n, runs):  # noqa: F811
    import torch
    lines = runs_of(n, runs, 7)
    order = torch.argsort(lines["nu0"], stable=True)
    got = []
    for ls in (lines, {k: v[order].contiguous() for k, v in lines.items()}):
        ctx.upload(ls)
        got.append(ctx.opacity(700.0, 0.5, 18.0, ("abs", 0.02), (0.0, 0.05, 60000)).clone())
    assert got[0].max().item() > 0 and torch.equal(got[0], got[1])


def test_cost(ctx):  # noqa: F811
    import time
    best = []
    for runs in (9, 17):
        lines = runs_of(400_000, runs, 5)
        ts = []
        for _ in range(20):
            t0 = time.perf_counter()
            ctx.upload(lines)
            ts.append(time.perf_counter() - t0)
        best.append(min(ts))
    assert best[0] < 0.9 * best[1], best
