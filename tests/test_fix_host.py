"""The block fixed-point transforms' own source (csrc/chanfs_fix.cuh), compiled for the host (no GPU):
its pass plans and twiddles for every supported length, and the error of its passes against extended
precision, beside that of the same passes in FP64."""

import ctypes
import os
import subprocess

import numpy as np
import pytest
from test_fix_layouts import radices, smooth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2502_06296_gb300", "csrc")
HARNESS = r"""
#include <cuda_runtime.h>
#include <complex>
#include <algorithm>
#include <cstring>
#include <vector>
using std::max;
using std::min;
#define CHANFS_FIX_ON_HOST
#define __noinline__
template <class To, class From> static To as(From f) { To t; memcpy(&t, &f, sizeof t); return t; }
static unsigned long long bits(double d) { return as<unsigned long long>(d); }
static int __double2hiint(double d) { return (int)(bits(d) >> 32); }
static int __double2loint(double d) { return (int)bits(d); }
static double __hiloint2double(int h, int l) {
  return as<double>(((unsigned long long)(unsigned)h << 32) | (unsigned)l);
}
static double __longlong_as_double(long long v) { return as<double>(v); }
static float __uint_as_float(unsigned u) { return as<float>(u); }
static unsigned __float_as_uint(float f) { return as<unsigned>(f); }
static unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
  return (unsigned)(((((unsigned long long)hi << 32) | lo) << (s & 31)) >> 32);
}
static unsigned __float2uint_ru(float f) { return (unsigned)ceilf(f); }
static int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
static double __ll2double_rn(long long v) { return (double)v; }
template <class T> static T __ldg(const T* p) { return *p; }
#include "chanfs_fix.cuh"
using namespace chanfs;

// One line through the first pass (as the kernels' first_pass), the middle passes and the last one.
template <bool PAIR, bool INV> static void run(int n, const double2* in, double2* out) {
  const int np = fix_npass<PAIR>(n);
  std::vector<int4> tw;
  const FixRoots roots(n);
  for (int p = 0; p < np; ++p) {
    const int R = fix_rad<PAIR, INV>(n, p), L = fix_span<PAIR, INV>(n, p);
    for (int r = 1; r < R; ++r)
      for (int k = 0; k < L; ++k) tw.push_back(roots.at((long long)r * k * (n / (L * R)), INV));
  }
  std::vector<Fix> a(n), b(n);
  FixScale f;
  const auto first = [&](auto rad) {
    constexpr int R = decltype(rad)::value;
    const int Q = n / R;
    unsigned top = 0, most = 0, quanta = 0;
    std::vector<float> sums;
    for (int j = 0; j < Q; ++j) {
      float sum = 0;
      for (int r = 0; r < R; ++r) fix_gather(in[j + r * Q], top, sum);
      most = max(most, __float_as_uint(sum));
      sums.push_back(sum);
    }
    if (fix_uses_sum<PAIR, INV>(n))
      for (float s : sums) quanta += fix_quanta(s, top, most);
    f = fix_scale_of(top, most, quanta, fix_growth<PAIR, INV>(n), 61, fix_div<PAIR, INV>(n, 1));
    for (int j = 0; j < Q; ++j) {
      Fix v[R];
      for (int r = 0; r < R; ++r) v[r] = fix_from(in[j + r * Q], f.s);
      fdft<R, INV>(v);
      for (int r = 0; r < R; ++r) a[j * R + r] = v[r];
    }
  };
  const auto pass = [&](auto rad, int p) {
    constexpr int R = decltype(rad)::value;
    const int L = fix_span<PAIR, INV>(n, p);
    const int4* w = tw.data() + fix_twoff<PAIR, INV>(n, p);
    const auto at = [](int e) { return e; };
    for (int j = 0; j < n / R; ++j)
      if (R == 3 && fix_halves<PAIR>(n)) fix_butterfly<3, INV, true>(a.data(), b.data(), j, n / R, L, w, at);
      else fix_butterfly<R, INV, false>(a.data(), b.data(), j, n / R, L, w, at);
    a.swap(b);
  };
  const auto by_radix = [&](int R, auto go) {
    if (R == 8) go(std::integral_constant<int, 8>{});
    else if (R == 6) go(std::integral_constant<int, 6>{});
    else if (R == 4) go(std::integral_constant<int, 4>{});
    else if (R == 3) go(std::integral_constant<int, 3>{});
    else go(std::integral_constant<int, 2>{});
  };
  by_radix(fix_rad<PAIR, INV>(n, 0), first);
  for (int p = 1; p < np; ++p) by_radix(fix_rad<PAIR, INV>(n, p), [&](auto r) { pass(r, p); });
  for (int e = 0; e < n; ++e) out[e] = fix_to(a[e], f.s - fix_drop<PAIR, INV>(n), f.kind);
}

// The same passes in floating point, products by tables rounded once.
template <class T> static void plain(int n, const int* rad, int inv, const double2* in, T* re, T* im) {
  using C = std::complex<T>;
  const long double tau = (inv ? 2 : -2) * 3.14159265358979323846264338327950288L;
  std::vector<C> a(n), b(n), w(n);
  for (int e = 0; e < n; ++e) {
    a[e] = C(in[e].x, in[e].y);
    w[e] = C((T)cosl(tau * e / n), (T)sinl(tau * e / n));
  }
  for (int p = 0, L = 1; p < 16 && rad[p]; L *= rad[p++]) {
    const int R = rad[p], Q = n / R;
    for (int j = 0; j < Q; ++j) {
      const int k = j % L;
      C v[8];
      for (int r = 0; r < R; ++r) v[r] = r * k ? a[j + r * Q] * w[r * k * (n / (L * R))] : a[j + r * Q];
      for (int q = 0; q < R; ++q) {
        C s = v[0];
        for (int r = 1; r < R; ++r) s += v[r] * w[(q * r % R) * Q];
        b[(j - k) * R + k + q * L] = s;
      }
    }
    a.swap(b);
  }
  for (int e = 0; e < n; ++e) {
    re[e] = a[e].real();
    im[e] = a[e].imag();
  }
}

extern "C" int passes(int n, int pair, int inv, int* rad, int* span, int* off) {
  int p = 0;
  for (; p < 16; ++p) {
    const int R = pair ? (inv ? fix_rad<true, true>(n, p) : fix_rad<true, false>(n, p)) : fix_rad<false, false>(n, p);
    rad[p] = p < fix_npass<true>(n) || !pair ? R : 0;
    if (!rad[p]) break;
    span[p] = pair && inv ? fix_span<true, true>(n, p) : pair ? fix_span<true, false>(n, p) : fix_span<false, false>(n, p);
    off[p] = pair && inv ? fix_twoff<true, true>(n, p) : pair ? fix_twoff<true, false>(n, p) : fix_twoff<false, false>(n, p);
  }
  return p;
}
extern "C" int halves(int n, int pair) { return pair ? fix_halves<true>(n) : fix_halves<false>(n); }
extern "C" void roots(int n, int conj, long double* re, long double* im) {
  const FixRoots w(n);
  for (int e = 0; e < n; ++e) {
    const int4 v = w.at(e, conj);
    re[e] = ldexpl((long double)v.x, -30) + ldexpl((long double)v.y, -62);
    im[e] = ldexpl((long double)v.z, -30) + ldexpl((long double)v.w, -62);
  }
}
// Squared errors of the fixed-point passes and of the FP64 ones, and the squared norm.
extern "C" void errors(int n, int pair, int inv, const double* in, double* got) {
  const double2* x = reinterpret_cast<const double2*>(in);
  std::vector<double2> y(n);
  int rad[17] = {}, s[17], o[17];
  passes(n, pair, inv, rad, s, o);
  if (pair && inv) run<true, true>(n, x, y.data());
  else if (pair) run<true, false>(n, x, y.data());
  else if (inv) run<false, true>(n, x, y.data());
  else run<false, false>(n, x, y.data());
  std::vector<long double> re(n), im(n);
  std::vector<double> dr(n), di(n);
  plain<long double>(n, rad, inv, x, re.data(), im.data());
  plain<double>(n, rad, inv, x, dr.data(), di.data());
  const auto sq = [](long double a, long double b) { return (double)(a * a + b * b); };
  for (int e = 0; e < n; ++e) {
    got[0] += sq(y[e].x - re[e], y[e].y - im[e]);
    got[1] += sq(dr[e] - re[e], di[e] - im[e]);
    got[2] += sq(re[e], im[e]);
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fix")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-w", "-ffp-contract=off", "-fPIC", "-shared", "-I", CSRC, "-I",
                    "/usr/local/cuda/include", "-o", str(d / "h.so"), str(d / "h.cpp")], check=True)
    return ctypes.CDLL(str(d / "h.so"))


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def columns(kind, n, rng):
    z = rng.standard_normal((6, n)) + 1j * rng.standard_normal((6, n))
    if kind == "spectrum":
        return z / np.maximum(np.minimum(np.arange(n), n - np.arange(n)), 0.5) ** 2
    if kind == "one value":
        z *= 1e-9
        z[np.arange(6), rng.integers(0, n, 6)] += 1.0
    if kind == "decades":
        z *= 10.0 ** rng.uniform(-6, 6, (6, n))
    return z


@pytest.mark.parametrize("n", smooth(9, 4096))
def test_plans_and_twiddles(lib, n):
    rad, span, off = (np.zeros(17, np.int32) for _ in range(3))
    for pair in (0, 1) if n <= 2048 else (0,):
        for inv in (0, 1):
            count = lib.passes(n, pair, inv, ptr(rad), ptr(span), ptr(off))
            want = radices(n, bool(pair))
            want = want[::-1] if pair and inv else want
            # the kernels whose radix-3 passes divide by 2 have these radices alone
            if lib.halves(n, pair):
                assert set(want) == {3, 6} or set(want) == {3}
                assert n % 81 == 0  # (none of them has a compiled kernel)
            L = np.cumprod([1] + want[:-1])
            assert 2 <= count <= 8 and list(rad[:count]) == want and list(span[:count]) == list(L)
            assert list(off[:count]) == list(np.cumsum([0] + [(r - 1) * l for r, l in zip(want, L)])[:-1])
    re, im = np.zeros(n, np.longdouble), np.zeros(n, np.longdouble)
    a = 2 * np.arccos(np.longdouble(-1)) * np.arange(n, dtype=np.longdouble) / n
    for conj in (0, 1):
        lib.roots(n, conj, ptr(re), ptr(im))
        # one place of 2^-62 (a low word of -2^31 moves by one), and the rounding of numpy's angle
        assert np.max(np.abs(re - np.cos(a))) <= 2.0**-62 + 8 * 2.0**-63
        assert np.max(np.abs(im + (1 - 2 * conj) * np.sin(a))) <= 2.0**-62 + 8 * 2.0**-63


@pytest.mark.parametrize("kind", ["spectrum", "one value", "white", "decades"])
@pytest.mark.parametrize("n", smooth(9, 4096))
def test_error_is_that_of_an_fp64_transform(lib, n, kind):
    """FP64 transforms stay within about 0.6 log2(n) 2^-53 of the exact one in L2 (numpy's; the plain FP64
    passes that `errors` runs beside the others are at 0.9 to 2.7), and so do these."""
    z = columns(kind, n, np.random.default_rng(n))
    for pair in (0, 1) if n <= 2048 else (0,):
        for inv in (0, 1):
            got = np.zeros(3)
            for col in z:
                lib.errors(n, pair, inv, ptr(np.ascontiguousarray(col)), ptr(got))
            assert np.sqrt(got[:2] / got[2]).max() * 2**53 < 0.6 * np.log2(n), (pair, inv)
