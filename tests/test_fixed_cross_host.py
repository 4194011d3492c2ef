"""The cross terms of a fixed-point sum in FP32 (fx_cross of csrc/fixed.cuh), compiled for the host, against the FMA chain
they take the place of: blocks of K steps of the orders' stencils, over windows whose values lie within kFxNear bits of the
tile's largest one.  Over 20000 windows of each kind neither the root mean square error nor the largest one, relative to
the exact sum, is above the chain's."""
import ctypes
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
// n taps w + low over `count` windows v; the tile's largest value has an exponent `up` above the window's own.
// err: squares' sum and largest of the chain, of the FP32 cross terms, relative to the exact sum (__float128).
extern "C" int cross(int n, const double *w, const double *low, int count, const double *v, int up, double *err) {
  FxTaps<31> t;
  fx_prepare(w, n, &t, low);
  if (!t.ok) return 0;
  for (int k = 0; k < count; ++k, v += n) {
    __float128 exact = 0;
    int mag = 0;
    for (int i = 0; i < n; ++i) {
      exact += ((__float128)w[i] + (__float128)low[i]) * (__float128)v[i];
      if (fx_mag(v[i]) > mag) mag = fx_mag(v[i]);
    }
    const int E = (mag >> 20) + up;
    double chain = w[n / 2] * v[n / 2];
    for (int i = 0; i < n; ++i) if (i != n / 2) chain = std::fma(w[i], v[i], chain);
    int64_t A = 0;
    FxCross c = {0.0f, 0.0f};
    for (int m = 0; m < n; ++m) {
      const int j = fx_inward(m, n);
      const Fx f = fx_split(fx_from(v[j], E));
      A = fx_mad(t.w1[j], f.hi, A);
      fx_cross(c, t, j, (float)f.lo, (float)f.hi);
    }
    const double got[2] = {chain, fx_to(fx_join_cross(A, c), E - 1023 - t.sw)};
    for (int g = 0; g < 2; ++g) {
      const double d = (double)(((__float128)got[g] - exact) / exact);
      err[2 * g] += d * d;
      if (std::fabs(d) > err[2 * g + 1]) err[2 * g + 1] = std::fabs(d);
    }
  }
  return 1;
}
extern "C" int near_bits() { return kFxNear; }
"""
CD1 = {2: [-1 / 2, 0.0, 1 / 2], 4: [1 / 12, -2 / 3, 0.0, 2 / 3, -1 / 12],
       6: [-1 / 60, 3 / 20, -3 / 4, 0.0, 3 / 4, -3 / 20, 1 / 60]}
CD2 = {2: [1.0, -2.0, 1.0], 4: [-1 / 12, 4 / 3, -5 / 2, 4 / 3, -1 / 12],
       6: [1 / 90, -3 / 20, 3 / 2, -49 / 18, 3 / 2, -3 / 20, 1 / 90]}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("cross")
    src = d / "cross.cpp"
    src.write_text(SRC)
    so = str(d / "cross.so")
    r = subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", ROOT, str(src), "-o", so],
                       capture_output=True, text=True)
    if r.returncode != 0 and "__float128" in r.stderr:
        pytest.skip("no __float128 on this machine")
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


@pytest.mark.parametrize("smooth", [True, False])
@pytest.mark.parametrize("r", [0.01, 0.02, 0.1])
@pytest.mark.parametrize("K", [2, 3, 4])
@pytest.mark.parametrize("order", [2, 4, 6])
def test_cross_terms_in_fp32_are_no_worse_than_the_chain(lib, order, K, r, smooth):
    if order == 6 and r > 0.02:
        pytest.skip("not a stable step")
    one = [Fraction(r * b - 0.003 * a) for a, b in zip(CD1[order], CD2[order])]
    one[order // 2] += 1
    taps = [Fraction(1)]
    for _ in range(K):
        nxt = [Fraction(0)] * (len(taps) + order)
        for i, a in enumerate(taps):
            for j, b in enumerate(one):
                nxt[i + j] += a * b
        taps = nxt
    n, count = len(taps), 20000
    w = np.array([float(t) for t in taps])
    low = np.array([float(t - Fraction(float(t))) for t in taps])
    rng = np.random.default_rng([order, K, int(1000 * r), smooth])
    x = np.arange(n) - n // 2
    base = 1.0 + 0.9 * rng.random((count, 1))
    if smooth:  # values that change by a ten-thousandth from cell to cell, down to the bottom of a binade
        v = np.where(rng.random((count, 1)) < 0.5, base, 1.0 + 1e-3 * rng.random((count, 1)))
        v = v * (1.0 + 2e-5 * x * rng.random((count, 1))) + 1e-7 * rng.random((count, n))
    else:
        v = base * (1.0 + 0.3 * (rng.random((count, n)) - 0.5))
    v = np.ascontiguousarray(v)
    D = ctypes.c_void_p
    for up in range(lib.near_bits() + 1):
        err = np.zeros(4)
        assert lib.cross(n, w.ctypes.data_as(D), low.ctypes.data_as(D), count, v.ctypes.data_as(D), up, err.ctypes.data_as(D))
        assert err[2] <= err[0] and err[3] <= err[1], (up, np.sqrt(err[[0, 2]] / count), err[[1, 3]])
