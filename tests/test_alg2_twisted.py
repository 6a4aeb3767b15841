"""The reduced system of Algorithm 2 factored from both ends
(csrc/chanfs_alg2.cuh, alg2_reduced_twisted), applied as the run-time kernel
does, against numpy (no GPU)."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2502_06296_gb300", "csrc")
HARNESS = """
#define __host__
#define __device__
#include "chanfs_alg2.cuh"
extern "C" void twisted(int J, const double* a, const double* b, const double* c, double* f) {
  chanfs::alg2_reduced_twisted<double>(J, a, b, c, f, f + J, f + 2 * J);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("twisted")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-I", CSRC, "-o", str(d / "h.so"),
                    str(d / "h.cpp")], check=True)
    return ctypes.CDLL(str(d / "h.so"))


@pytest.mark.parametrize("J", [2, 4, 6, 24, 32, 128])
@pytest.mark.parametrize("margin", [1.0001, 2.0, 1e6])
def test_twisted_factors_solve_the_reduced_system(lib, J, margin):
    rng = np.random.default_rng(J)
    a, c = -rng.random(J), -rng.random(J)
    a[0] = c[-1] = 0.0
    b = margin * (np.abs(a) + np.abs(c)) + 1e-3
    f = np.zeros((3, J))
    p = lambda x: x.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
    lib.twisted(J, p(a), p(b), p(c), p(f))
    rl, rip, ripc = f
    d = rng.standard_normal(J)
    h, y, x = J // 2, d.copy(), np.empty(J)
    for j in range(1, h):
        y[j] -= rl[j] * y[j - 1]
    for j in range(J - 2, h - 1, -1):
        y[j] -= rl[j] * y[j + 1]
    x[h - 1] = rip[h - 1] * y[h - 1] - ripc[h - 1] * y[h]
    x[h] = rip[h] * y[h] - ripc[h] * y[h - 1]
    for j in range(h - 2, -1, -1):
        x[j] = rip[j] * y[j] - ripc[j] * x[j + 1]
    for j in range(h + 1, J):
        x[j] = rip[j] * y[j] - ripc[j] * x[j - 1]
    M = np.diag(b) + np.diag(a[1:], -1) + np.diag(c[:-1], 1)
    # backward error of a stable elimination: J roundings of 2^-53 each, a few per row
    assert np.max(np.abs(M @ x - d)) < 8 * J * 2.0**-53 * np.max(np.abs(M) @ np.abs(x) + np.abs(d))


@pytest.mark.parametrize("J", [2, 4, 32])
@pytest.mark.parametrize("e", [-900, -600, 600, 1000])
def test_twisted_factors_follow_a_power_of_two(lib, J, e):
    """Rows times 2^e (coefficients c / dz^2 of any size): multipliers unchanged, inverse pivots and the two middle
    rows, which multiply right-hand sides, times 2^-e."""
    rng = np.random.default_rng(J)
    a, c = -rng.random(J), -rng.random(J)
    a[0] = c[-1] = 0.0
    b = 1.5 * (np.abs(a) + np.abs(c)) + 1e-3
    p = lambda x: x.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
    f, g = np.zeros((3, J)), np.zeros((3, J))
    lib.twisted(J, p(a), p(b), p(c), p(f))
    s = [np.ldexp(x, e) for x in (a, b, c)]
    lib.twisted(J, *map(p, s), p(g))
    f[1] = np.ldexp(f[1], -e)
    f[2, J // 2 - 1 : J // 2 + 1] = np.ldexp(f[2, J // 2 - 1 : J // 2 + 1], -e)
    assert np.isfinite(g).all() and np.array_equal(g, f)
