"""Which core kernel of the FP32 form a call takes (core_nodes_possible of route.cuh,
compiled for the host): the one with nodes whenever a line of the list can have a beta
small enough, the other on the grids where none can, with masses per line too."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1503_03806_gb300", "csrc")
SRC = r"""
#include "route.cuh"
extern "C" int possible(double nu_min, double dnu, int64_t n, double kc, double mass_min) {
  return helk::core_nodes_possible(nu_min, dnu, n, kc, mass_min);
}
extern "C" double beta_max() { return helk::CORE_NODE_BETA; }
"""
D, I = ctypes.c_double, ctypes.c_int64


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("core")
    (d / "c.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "c.cpp"), "-o", str(d / "c.so")],
                   check=True)
    so = ctypes.CDLL(str(d / "c.so"))
    so.beta_max.restype = D
    return so


def kc(T, mass):
    return np.sqrt(np.log(2.0)) / (np.sqrt(2.0 * np.log(2.0) * 1.380649e-16 * T / (mass * 1.66053906660e-24)) / 2.99792458e10)


def test_never_without_a_line_that_needs_it(lib):
    rng = np.random.default_rng(4)
    found = [0, 0]
    for _ in range(3000):
        T, dnu = 10.0 ** rng.uniform(1.5, 3.8), 10.0 ** rng.uniform(-4, 1)
        n, nu_min = int(10.0 ** rng.uniform(1, 6)), rng.choice([0.0, 500.0, 12000.0])
        masses = rng.choice([1.0, 2.0, 18.0, 44.0, 300.0], rng.integers(1, 4))
        nu = rng.uniform(max(nu_min, dnu), nu_min + n * dnu * 1.001, 50)
        beta = dnu * kc(T, rng.choice(masses, 50)) / nu
        p = lib.possible(D(nu_min), D(dnu), I(n), D(kc(T, 1.0)), D(masses.min()))
        found[p] += 1
        assert p or beta.min() > lib.beta_max()
    assert min(found) > 0


@pytest.mark.parametrize("dnu,n,masses,want", [(0.01, 3_000_000, (16.0, 18.0, 44.0), 0), (0.1, 300_000, (2.0, 18.0), 0),
                                               (0.001, 30_000_000, (16.0, 18.0, 44.0), 1)])
def test_lists_with_masses(lib, dnu, n, masses, want):
    assert lib.possible(D(0.0), D(dnu), I(n), D(kc(1500.0, 1.0)), D(min(masses))) == want
