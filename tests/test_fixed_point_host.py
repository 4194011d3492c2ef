"""The block fixed-point arithmetic of csrc/fixed.cuh, compiled for the host, against exact rational sums.

A sum of n products must come out within half a unit in the last place of the exact value plus the representation's
own error, which is below 2^-58 of (largest value) x (sum of the weights' magnitudes): values are cut at 2^-61 of the
largest one's binade (one unit each, so at most sum |w|), the weights are rounded at 2^-60 / 1.9 of their sum, the low by
low products left out are below 2^-60 in all, and the joins round three times at 2^-61.  With the cross terms in FP32
the bound is (2 n + 4) roundings of 2^-24 on terms below 2^-31 of the same product."""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "paper_1702_00496_gb300/csrc/fixed.cuh"
#include <cmath>
using namespace atfd;
extern "C" int fx_sum(int n, const double *w, const double *v, int f32, double *out) {
  FxTaps<31> t;
  fx_prepare(w, n, &t);
  int mag = 0;
  for (int i = 0; i < n; ++i) if (fx_mag(v[i]) > mag) mag = fx_mag(v[i]);
  const int E = mag >> 20;
  if (!t.ok || !fx_usable(E)) return 0;
  int64_t A = 0, B = kFxB0, C = kFxC0;
  float c = 0.0f;
  for (int i = 0; i < n; ++i) {
    const Fx f = fx_split(fx_from(v[i], E));
    A = fx_mad(t.w1[i], f.hi, A);
    B = fx_mad(t.w1[i], f.lo, B);
    C = fx_mad(t.w0[i], f.hi, C);
    c = std::fma(t.f1[i], (float)f.lo, c);
    c = std::fma(t.f0[i], (float)f.hi, c);
  }
  const int64_t R = f32 ? A + (int64_t)std::lrintf(c) * 8 : fx_join(A, B, C);
  *out = fx_to(R, E - 1023 - t.sw);
  return 1;
}
extern "C" int fx_weights(int n, const double *w, const double *low, int64_t *W) {
  FxTaps<31> t;
  fx_prepare(w, n, &t, low);
  for (int i = 0; i < n; ++i) W[i] = (int64_t)t.w1[i] * (1ll << kFxLowBits) + t.w0[i];
  return t.sw;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    src = d / "fx.cpp"
    src.write_text(SRC)
    so = str(d / "fx.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", ROOT, str(src), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


def _sum(lib, w, v, f32):
    out = ctypes.c_double()
    n = len(w)
    D = ctypes.c_double * n
    ok = lib.fx_sum(n, D(*w), D(*v), int(f32), ctypes.byref(out))
    return out.value if ok else None


def _weights(rng, n, kind):
    if kind == "stencil":  # a second difference and a first one, like the merged taps
        w = rng.uniform(-1, 1, n) * 0.5 ** np.abs(np.arange(n) - n // 2)
    elif kind == "ones":
        w = np.full(n, 1.0 / n)
    else:
        w = rng.uniform(-1, 1, n) * 2.0 ** rng.integers(-40, 40)
    return w


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("n", [1, 3, 5, 7, 17, 25, 31])
@pytest.mark.parametrize("kind", ["stencil", "ones", "any"])
def test_sums_against_exact_rationals(lib, n, kind, f32):
    rng = np.random.default_rng([n, len(kind), f32])
    for trial in range(200):
        w = _weights(rng, n, kind)
        scale = 2.0 ** rng.integers(-200, 200)
        v = rng.uniform(-1, 1, n) * scale * 2.0 ** rng.integers(-12, 1, n)
        if trial % 3 == 0:
            v = scale * (1.0 + 1e-6 * rng.uniform(-1, 1, n))
        if trial % 7 == 0:  # the ends of a binade, exact powers, zeros of both signs
            v = scale * rng.choice([1.0, -1.0, math.nextafter(2.0, 0.0), -math.nextafter(2.0, 0.0), 0.0, -0.0, 2.0 ** -70], n)
            v[rng.integers(n)] = scale
        got = _sum(lib, list(w), list(v), f32)
        assert got is not None
        exact = sum((Fraction(a) * Fraction(b) for a, b in zip(w.tolist(), v.tolist())), Fraction(0))
        size = Fraction(float(np.abs(v).max())) * Fraction(float(np.abs(w).sum()))
        rep = size * Fraction(2 * n + 4, 2 ** 55) if f32 else size / 2 ** 58
        ulp = Fraction(math.ulp(abs(float(exact)))) if exact else Fraction(0)
        assert abs(Fraction(got) - exact) <= rep + ulp / 2 + (Fraction(math.ulp(got)) / 2 if got else 0)


@pytest.mark.parametrize("low", [False, True])
@pytest.mark.parametrize("n", [1, 17, 25])
def test_weights_hold_the_low_parts_too(lib, n, low):
    """Weights given as a double and what lies below its last bit come out as the nearest whole number of 2^-sw (and one
    more rounding of 2^-53 of the part below a unit)."""
    rng = np.random.default_rng([n, low])
    for kind in ("stencil", "ones", "any"):
        w = _weights(rng, n, kind)
        wl = np.abs(w) * 2.0 ** -53 * rng.uniform(-1, 1, n)
        W = (ctypes.c_int64 * n)()
        D = ctypes.c_double * n
        sw = lib.fx_weights(n, D(*w), D(*wl) if low else None, W)
        for a, b, c in zip(w.tolist(), wl.tolist(), W):
            exact = (Fraction(a) + (Fraction(b) if low else 0)) * 2 ** sw
            assert abs(c - exact) <= Fraction(1, 2) + Fraction(1, 2 ** 40)


def test_what_is_not_summed(lib):
    """Infinities, NaN, values at the ends of the exponent range and weights that cannot be scaled are refused."""
    for v in ([math.inf, 1.0, 1.0], [math.nan, 1.0, 1.0], [0.0, 0.0, 0.0], [1e-290, 0.0, 0.0], [1e300, 1.0, 1.0]):
        assert _sum(lib, [0.25, 0.5, 0.25], v, False) is None
    for w in ([math.inf, 1.0, 1.0], [math.nan, 1.0, 1.0], [0.0, 0.0, 0.0], [1e30, 1.0, 1.0], [1e-30, 0.0, 0.0]):
        assert _sum(lib, w, [1.0, 2.0, 3.0], False) is None
    assert _sum(lib, [0.5, 0.0, -0.5], [3.0, 7.0, 3.0], False) == 0.0


def test_division_by_multiplication():
    """fast_div / fdiv of internal.h: the quotient for every divisor kind and numerators up to 2^30, in Python's integers."""
    rng = np.random.default_rng(3)
    divisors = [1, 2, 3, 4, 5, 7, 8, 14, 16, 62, 1022, 1024, 1023, 4097, 2 ** 20 - 1, 2 ** 28, 2 ** 28 + 1, 2 ** 30 - 1]
    divisors += [int(v) for v in rng.integers(1, 2 ** 30, 400)]
    for d in divisors:
        s = 0
        while (4 << s) < d:
            s += 1
        m = ((1 << (32 + s)) + d - 1) // d
        assert m <= 2 ** 32 and (m < 2 ** 32 or d == 1)
        ns = [0, 1, d - 1, d, d + 1, 2 ** 30 - 1, (2 ** 30 - 1) // d * d, (2 ** 30 - 1) // d * d - 1]
        ns += [int(v) for v in rng.integers(0, 2 ** 30, 50)]
        for n in ns:
            if 0 <= n < 2 ** 30:
                assert (n if d == 1 else (n * m >> 32) >> s) == n // d, (n, d)
