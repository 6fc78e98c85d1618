"""FP64 opacity under a Lorentz cutoff, whose windows follow the condition: low
pressures take the point-by-point kernels whatever the cap, and a batch over
pressures takes both routes.  Each condition against the counting call at 1e-9, and
the batch against single calls bit for bit: list fields that decide the width, chunks
under a small budget, replays with other conditions and another share of them on each
route.  The cost of a low-pressure call is at most that of the counting call and a
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


def lines_of(fields):
    lines = synth.random_lines(4000, 9, 3000.0, 3300.0, with_elower=True)
    rng = np.random.default_rng(2)
    if "self" in fields:
        lines["gamma_self"] = rng.uniform(0.0, 3.0, 4000)
    if "ncoll" in fields:
        lines["n_coll"] = rng.uniform(-0.5, 1.2, 4000)
    if "zero" in fields:
        lines["gamma_air"][:] = 0.0
    return lines


P_MIX = [1e-8, 3.0, 1e-5, 0.3, 1e-3, 1e-7, 0.0, 10.0, 1e-4, 0.03, 1e-6]


@pytest.mark.parametrize("fields", [(), ("self",), ("ncoll",), ("self", "ncoll"), ("zero",), ("zero", "self")])
@pytest.mark.parametrize("cut", [("lorentz", 500.0, 100.0), ("lorentz", 500.0, 0.2), ("lorentz", 20.0, 5.0)])
def test_mixed_batch(ctx, fields, cut):
    ctx.upload(lines_of(fields))
    grid = (3000.0, 0.01, 30_000)
    T = np.linspace(250.0, 2800.0, len(P_MIX))
    kb = ctx.opacity_batch(T, P_MIX, 18.0, cut, grid).cpu().numpy()
    ev, _ = ctx.batch_stats(len(P_MIX))
    for k, (t, p) in enumerate(zip(T, P_MIX)):
        one = ctx.opacity(t, p, 18.0, cut, grid).cpu().numpy()
        assert ctx.stats()[0] == ev[k]
        assert np.array_equal(one, kb[k]), (t, p)
        ref = ctx.opacity(t, p, 18.0, cut, grid, count_regions=True).cpu().numpy()
        assert np.array_equal(one != 0, ref != 0), (t, p)
        np.testing.assert_allclose(one, ref, rtol=1e-9)


def test_replays_and_chunks(ctx):
    ctx.upload(lines_of(("self",)))
    grid, cut = (3000.0, 0.01, 30_000), ("lorentz", 500.0, 100.0)
    rng = np.random.default_rng(0)
    try:
        for budget in (0, 3 * (4000 * 96 + 30_000 * 8), 1):
            ctx.set_batch_budget(budget)
            for _ in range(4):
                P = rng.permutation(P_MIX)
                if rng.random() < 0.5:
                    P[:4] = 1.0
                T = rng.uniform(300.0, 2500.0, len(P))
                kb = ctx.opacity_batch(T, P, 18.0, cut, grid, accumulate=False).cpu().numpy()
                for k in range(len(P)):
                    assert np.array_equal(kb[k], ctx.opacity(T[k], P[k], 18.0, cut, grid).cpu().numpy()), (budget, k)
    finally:
        ctx.set_batch_budget(0)


@pytest.mark.parametrize("P", [1e-7, 1e-5])
def test_cost(ctx, P):
    import torch
    ctx.upload(synth.random_lines(100_000, 5, 1.0, 30_000.0))
    out = torch.empty(3_000_000, dtype=torch.float64, device="cuda")
    best = []
    for count in (False, True):
        ms = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ctx.opacity(1500.0, P, 18.0, ("lorentz", 500.0, 100.0), (0.0, 0.01, 3_000_000), out=out, count_regions=count)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        best.append(min(ms))
    assert best[0] < 1.1 * best[1], best
