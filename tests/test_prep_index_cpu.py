"""The integer window bounds of the FP32 form's line preparation (prep_index of
k_lines.cu, the source itself compiled for the host): equal to ceil(v / dnu) and
floor(v / dnu), also where v is 0 (a window that begins or ends exactly on the
grid's first point), where the quotient is an integer or next to one, and where
it is too small for FP64 or too large for an index."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1503_03806_gb300", "csrc")

SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#include <algorithm>
using std::fmin;
#define __device__
#define __forceinline__ inline
#define __noinline__
static int __double2hiint(double v) { int64_t b; std::memcpy(&b, &v, 8); return (int)(b >> 32); }
static int __double2loint(double v) { int64_t b; std::memcpy(&b, &v, 8); return (int)b; }
%s
extern "C" void bounds(int64_t n, const double *v, const double *dnu, int *up, int *down) {
  for (int64_t i = 0; i < n; ++i) {
    up[i] = prep_index<true>(v[i], dnu[i], 1.0 / dnu[i]);
    down[i] = prep_index<false>(v[i], dnu[i], 1.0 / dnu[i]);
  }
}
"""


@pytest.fixture(scope="module")
def bounds(tmp_path_factory):
    src = open(os.path.join(CSRC, "k_lines.cu")).read()
    body = src[src.index("constexpr double PREP_MAGIC"):src.index("// The FP32 records with strengths as a mantissa")]
    d = tmp_path_factory.mktemp("prep")
    (d / "p.cpp").write_text(SHIM % body)
    so = str(d / "p.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", str(d / "p.cpp"), "-o", so],
                   check=True)
    lib = ctypes.CDLL(so)

    def run(v, dnu):
        v, dnu = np.broadcast_arrays(np.asarray(v, np.float64), np.asarray(dnu, np.float64))
        v, dnu = np.ascontiguousarray(v), np.ascontiguousarray(dnu)
        up, down = np.zeros(v.size, np.int32), np.zeros(v.size, np.int32)
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        lib.bounds(ctypes.c_int64(v.size), p(v), p(dnu), p(up), p(down))
        q = v / dnu
        clip = lambda x: np.clip(x, -2.0 ** 30, 2.0 ** 31 - 1).astype(np.int64)
        bad = (up != clip(np.ceil(q))) | (down != clip(np.floor(q)))
        assert not bad.any(), (v[bad][:5], dnu[bad][:5], up[bad][:5], down[bad][:5])

    return run


@pytest.mark.parametrize("v", [0.0, -0.0])
def test_zero(bounds, v):
    bounds(v, [1e-4, 0.01, 1.0 / 128, 0.3, 1.0, 5.0, 1e6])


def test_tiny_and_large(bounds):
    for v in (5e-324, 1e-310, 2.3e-308, 1e-300, 1e-20, 1e-9, 0.3, 1.0, 1e9, 1.07374e9, 1e15, 1e300):
        for s in (1.0, -1.0):
            bounds(s * v, [1e-4, 0.01, 1.0, 1e6])


def test_integers_and_neighbours(bounds):
    rng = np.random.default_rng(1)
    for dnu in (1e-4, 0.001, 0.01, 1.0 / 128, 0.3, 5.0):
        k = np.concatenate([np.arange(-300, 301), rng.integers(-2 ** 30, 2 ** 30, 20000)]).astype(float)
        v = k * dnu
        for w in (v, np.nextafter(v, np.inf), np.nextafter(v, -np.inf), v * (1 + 1e-15), v + 0.5 * dnu):
            bounds(w, dnu)
    bounds(rng.uniform(-1e4, 1e4, 100000), 10.0 ** rng.uniform(-4, 1, 100000))
