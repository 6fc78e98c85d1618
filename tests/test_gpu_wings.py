"""The interpolated-wings route of the opacity stage (lines taken on whole
panels of the grid through Chebyshev nodes) against the oracle's point-by-
point sums: grids at the edges of leaves (32 points), warp panels (128),
groups (1024) and coarser levels, windows from narrower than a panel to the
whole grid, broad and narrow lines, centres on and off the grid.

FP64 form: 1e-9 at every point.  FP32 form: the stated bar of the form, 1e-5
where the opacity exceeds 1e-8 of the maximum.  A line lost or taken twice on
one panel is off by the order of its own share.
"""
import numpy as np
import pytest

import oracle
from paper_1503_03806_gb300 import synth
from tests.helpers import NTHREADS, Case, assert_rel

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


def check(ctx, lines, case):
    from paper_1503_03806_gb300 import helk
    ctx.upload(lines)
    ko, _, _ = oracle.opacity(lines, case.oracle_cond(), nthreads=NTHREADS)
    assert_rel(case.gpu(ctx).cpu().numpy(), ko, 1e-9, "FP64")
    k32 = case.gpu(ctx, precision=helk.HELK_PREC_F32_KAHAN).cpu().numpy()
    ctx.sync()
    sel = ko > 1e-8 * ko.max()
    assert np.all(np.isfinite(k32)) and np.max(np.abs(k32[sel] - ko[sel]) / ko[sel]) <= 1e-5


@pytest.mark.parametrize("n", [1, 31, 32, 33, 127, 129, 1023, 1024, 1025, 8191, 8193, 66_000])
@pytest.mark.parametrize("cut", [("abs", 1.0), ("abs", 12.0), ("lorentz", 500.0, 40.0), ("none",)])
def test_panel_edges(ctx, n, cut):
    hi = 100.0 + 0.01 * n
    lines = synth.random_lines(60, 31 + n, 99.0, hi + 1.0)
    check(ctx, lines, Case(1500.0, 1.0, 18.0, (100.0, 0.01, n), cut))


@pytest.mark.parametrize("P", [1e-4, 0.3, 20.0, 3000.0])
@pytest.mark.parametrize("nu", [50.0, 20000.0])
def test_line_shapes(ctx, P, nu):
    # Doppler- to pressure-broadened, on a coarse and a fine grid in Doppler units
    lines = synth.random_lines(250, 77, nu, nu + 60.0, with_elower=True, extra_fields=True)
    check(ctx, lines, Case(900.0, P, 28.0, (nu, 0.003, 20_000 + 11), ("lorentz", 500.0, 25.0), q_ratio=0.4))


def test_dense_list_takes_several_batches(ctx):
    # more lines than a group's batch in shared memory, all of them near
    lines = synth.random_lines(6000, 78, 500.0, 520.0)
    check(ctx, lines, Case(700.0, 0.5, 18.0, (500.0, 0.01, 2000), ("abs", 8.0)))


@pytest.mark.parametrize("dnu,nu", [(1e-6, 800.0), (5.0, 1.0)])
def test_method_boundaries_on_extreme_grids(ctx, dnu, nu):
    # thousands of grid points in a Doppler unit, and thousands of Doppler units
    # between two points (a method changes from one point to the next)
    lines = synth.random_lines(40, 80, nu, nu + 3000 * dnu, extra_fields=True)
    check(ctx, lines, Case(1500.0, 0.1, 18.0, (nu - 20 * dnu, dnu, 3000), ("none",)))


def test_accumulate_and_weight(ctx):
    import torch
    from paper_1503_03806_gb300 import helk
    lines = synth.random_lines(200, 79, 0.0, 40.0)
    case = Case(1500.0, 1.0, 18.0, (0.0, 0.01, 4000 + 9), ("abs", 10.0))
    ctx.upload(lines)
    out = torch.full((case.grid[2],), 3e-22, dtype=torch.float64, device="cuda")
    case.gpu(ctx, out=out, precision=helk.HELK_PREC_F32_KAHAN, accumulate=True, weight=-0.5)
    ko, _, _ = oracle.opacity(lines, case.oracle_cond(), weight=1.0)
    assert np.max(np.abs(out.cpu().numpy() - (3e-22 - 0.5 * ko)) / (3e-22 + 0.5 * ko)) <= 1e-5
