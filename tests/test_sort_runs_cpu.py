"""The places of a merged line list (merged_place of sort_runs.cuh, compiled for
the host) at list lengths up to the longest accepted, 2^31 - 2 lines, whose indices
add up beyond 32 bits.  The centres are given by a formula of the index, so no list
is held; every read is checked to lie in the list.  Small lists against a stable
sort."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1503_03806_gb300", "csrc")

SRC = r"""
#define __host__
#define __device__
#define __forceinline__ inline
#include "sort_runs.cuh"
// Runs of equal length n / runs, element i of run r at i * runs + r (all distinct):
// element i of run r has the place i * runs + r.
extern "C" int64_t formula(int64_t n, int runs, int64_t l, int *outside) {
  helk::SortRuns R{};
  R.n = runs;
  const int64_t len = n / runs;
  for (int r = 0; r < runs; ++r) R.end[r] = (int)(len * (r + 1));
  return helk::merged_place(R, l, [=](int64_t i) {
    if (i < 0 || i >= n) *outside = 1;
    return (double)((i % len) * runs + i / len);
  });
}
extern "C" void places(int n, const double *nu0, int runs, const int *end, int64_t *at) {
  helk::SortRuns R{};
  R.n = runs;
  for (int r = 0; r < runs; ++r) R.end[r] = end[r];
  for (int l = 0; l < n; ++l) at[l] = helk::merged_place(R, l, [=](int64_t i) { return nu0[i]; });
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("runs")
    (d / "r.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "r.cpp"), "-o", str(d / "r.so")],
                   check=True)
    so = ctypes.CDLL(str(d / "r.so"))
    so.formula.restype = ctypes.c_int64
    return so


@pytest.mark.parametrize("runs", [2, 3, 16])
@pytest.mark.parametrize("n", [960, 2 ** 30 - 64, 2 ** 30 + 64, 2 ** 31 - 2])
def test_long_lists(lib, n, runs):
    n -= n % runs
    length = n // runs
    rng = np.random.default_rng(runs)
    ls = [0, 1, length - 1, length, n - length - 1, n - length, n - 2, n - 1] + [int(v) for v in rng.integers(0, n, 200)]
    for l in ls:
        outside = ctypes.c_int(0)
        at = lib.formula(ctypes.c_int64(n), runs, ctypes.c_int64(l), ctypes.byref(outside))
        assert outside.value == 0, (n, l)
        assert at == (l % length) * runs + l // length, (n, l)


def test_stable_order(lib):
    rng = np.random.default_rng(3)
    for runs in (1, 2, 5, 16):
        parts = [np.sort(rng.integers(0, 40, rng.integers(1, 50)).astype(float)) for _ in range(runs)]
        nu = np.concatenate(parts)
        end = np.cumsum([p.size for p in parts]).astype(np.int32)
        at = np.zeros(nu.size, np.int64)
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        lib.places(nu.size, p(nu), runs, p(end), p(at))
        want = np.empty(nu.size, np.int64)
        want[np.argsort(nu, kind="stable")] = np.arange(nu.size)
        assert np.array_equal(at, want)
