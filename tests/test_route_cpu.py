"""The rules that choose between interpolated wings and point-by-point sums
(route.cuh, compiled for the host): the number of lines near a stretch of the grid
against a count, and each form's rule on the faster side of the measured cases that
it states."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1503_03806_gb300", "csrc")

SRC = r"""
#include "route.cuh"
static helk::ListShape shape(int64_t n, const double *at) {
  helk::ListShape L{};
  L.n = n;
  for (int i = 0; i <= helk::LIST_CUTS; ++i) L.at[i] = at[i];
  return L;
}
extern "C" int cuts() { return helk::LIST_CUTS; }
extern "C" double near(int64_t n, const double *at, double nu_min, double dnu, int64_t ng, double points, double reach) {
  return helk::lines_near(shape(n, at), nu_min, dnu, ng, points, reach);
}
extern "C" int pay64(int64_t n, const double *at, double nu_min, double dnu, int64_t ng, double half,
                     double most) {
  return helk::wings_pay64(shape(n, at), nu_min, dnu, ng, most, half);
}
extern "C" int pay32(int64_t n, const double *at, double nu_min, double dnu, int64_t ng, double most) {
  return helk::wings_pay32(shape(n, at), nu_min, dnu, ng, most, 152);
}
"""
D, I = ctypes.c_double, ctypes.c_int64


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("route")
    (d / "r.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "r.cpp"), "-o", str(d / "r.so")],
                   check=True)
    so = ctypes.CDLL(str(d / "r.so"))
    so.near.restype = D
    return so


def at(lib, nu):
    c = lib.cuts()
    n = len(nu)
    a = np.ascontiguousarray(nu[[(n - 1) * i // c for i in range(c + 1)]])
    return a, a.ctypes.data_as(ctypes.c_void_p)


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 1000, 100_000])
@pytest.mark.parametrize("lo,hi", [(0.0, 300.0), (100.0, 130.0), (5000.0, 6000.0)])
def test_lines_near(lib, n, lo, hi):
    rng = np.random.default_rng(n)
    nu = np.sort(rng.uniform(lo, hi, n))
    a, p = at(lib, nu)
    for points, reach in ((2048.0, 30.0), (2048.0, 2500.0), (1.0, 100.0), (1e9, 0.0)):
        got = lib.near(I(n), p, D(0.0), D(0.01), I(30000), D(points), D(reach))
        w = 0.5 * min(points, 30000.0)
        want = 0.0
        for k in range(8):
            mid = w + (30000.0 - 2 * w) * (k + 0.5) / 8
            x0, x1 = (mid - w - reach) * 0.01, (mid + w + reach) * 0.01
            want += ((nu > x0) & (nu <= x1)).sum() / 8.0
        assert abs(got - want) <= 2.0 + 2.0 * n / lib.cuts(), (points, reach, got, want)


@pytest.mark.parametrize("n,nlines,half,wings", [
    (3_000_000, 1, 30, False), (3_000_000, 100, 25000, False), (3_000_000, 1000, 2500, False),
    (3_000_000, 1000, 25000, True), (3_000_000, 10_000, 30, True), (3_000_000, 100_000, 24, True),
    (3_000_000, 100_000, 23, False), (300_000, 100, 2500, False), (300_000, 1000, 30, True),
    (300_000, 100, 25000, True), (30_000, 300, 30, False), (3000, 30, 250, False), (30_000, 1000, 250, True),
    (30_000, 100, 250, False), (30_000, 10, 25000, False), (30_000, 100, 25000, True),
    (30_000, 10_000, 30, True), (3000, 10, 2500, False), (3000, 100, 250, True), (300, 10, 250, False),
    (300, 100, 30, True), (10_000, 300, 2000, True), (20_000, 3000, 24, True)])
def test_measured_cases(lib, n, nlines, half, wings):
    nu = np.sort(np.random.default_rng(1).uniform(0.05, n * 0.01, nlines))
    a, p = at(lib, nu)
    assert bool(lib.pay64(I(nlines), p, D(0.0), D(0.01), I(n), D(half), D(half))) == wings


@pytest.mark.parametrize("n,nlines,half,wings", [
    (3_000_000, 100_000, 2.2e-4, False), (3_000_000, 1_000_000, 2.2e-4, False), (3_000_000, 100_000, 0.022, False),
    (3_000_000, 1_000_000, 0.022, True), (3_000_000, 100_000, 0.22, True), (3_000_000, 100_000, 22.0, True),
    (300_000, 10_000, 0.022, False), (300_000, 10_000, 0.22, True), (30_000, 1000, 0.022, False),
    (30_000, 1000, 0.22, True), (30_000, 1000, 0.0, False)])
def test_measured_pressures(lib, n, nlines, half, wings):
    nu = np.sort(np.random.default_rng(1).uniform(0.05, n * 0.01, nlines))
    a, p = at(lib, nu)
    assert bool(lib.pay64(I(nlines), p, D(0.0), D(0.01), I(n), D(half), D(10000.0))) == wings


@pytest.mark.parametrize("n,nlines,half,wings", [
    (3000, 10, 2500, False), (3000, 30, 2500, False), (3000, 1000, 250, True), (3000, 10_000, 63, False),
    (30_000, 100, 2500, False), (30_000, 300, 25_000, True), (30_000, 1000, 2500, True), (30_000, 30, 25_000, False),
    (300_000, 3000, 2500, False), (300_000, 1000, 25_000, False), (300_000, 3000, 25_000, True),
    (300_000, 100_000, 250, True), (3_000_000, 3000, 25_000, False), (3_000_000, 100_000, 250, False),
    (3_000_000, 10_000, 25_000, True), (3_000_000, 100_000, 2500, True), (3_000_000, 1_000_000, 64, True)])
def test_measured_cases32(lib, n, nlines, half, wings):
    nu = np.sort(np.random.default_rng(1).uniform(0.05, n * 0.01, nlines))
    a, p = at(lib, nu)
    assert bool(lib.pay32(I(nlines), p, D(0.0), D(0.01), I(n), D(half))) == wings


def test_a_band_of_a_long_list32(lib):
    for nlines, wings in ((10_000, False), (1_000_000, True)):
        nu = np.sort(np.random.default_rng(1).uniform(0.05, 30000.0, nlines))
        a, p = at(lib, nu)
        assert bool(lib.pay32(I(nlines), p, D(10000.0), D(0.01), I(300_000), D(2500.0))) == wings


def test_lines_elsewhere_do_not_count(lib):
    nu = np.sort(np.random.default_rng(1).uniform(0.05, 30000.0, 10_000))
    a, p = at(lib, nu)
    assert not lib.pay64(I(10_000), p, D(10000.0), D(0.01), I(3000), D(100.0), D(100.0))
    nu = np.sort(np.random.default_rng(1).uniform(20000.0, 30000.0, 1_000_000))
    a, p = at(lib, nu)
    assert not lib.pay64(I(1_000_000), p, D(0.0), D(0.01), I(300_000), D(2500.0), D(2500.0))
