"""The scale of the tiles' ring of planes (FxRing of csrc/fixed.cuh), compiled for the host: planes are laid down one by
one as the 3D step's march lays them, outputs are summed along z from the ring's entries, and an output that the rule lets
through (its own value at least fx_least of 10 bits) must be good to a few ulp of the largest value of its own stencil.

In units of 2^-62 of the scale such a value is 2^52 2^lift at least.  The sum may be off by 2^lift for the cut entries, by
half a unit per tap for the products left out and by two for the joins (a unit of the sum is two at most where the weights
sum to one), so by (6 + n) 2^-53 of that value, and the result's rounding is one more."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "paper_1702_00496_gb300/csrc/fixed.cuh"
#include <vector>
using namespace atfd;
// np planes of w cells; out[o][c]: the sum of cell c over planes o-H .. o+H, fixed[o][c]: let through
extern "C" int march(int np, int w, const double *v, int H, const double *wt, double *out, unsigned char *fixed) {
  FxTaps<31> t;
  fx_prepare(wt, 2 * H + 1, &t);
  if (!t.ok) return 0;
  const int NR = 2 * H + 2;
  std::vector<int64_t> ring((size_t)NR * w, 0);
  FxRing scale;
  FxPlanes planes = {};
  for (int i = 0; i < np + 2; ++i) {
    const int o = i - 2 - H;
    if (o >= H) {
      const int lift = fx_ring_lift(scale, planes, o, H);
      const bool usable = lift <= kFxLift && scale.E >= 0;
      for (int c = 0; c < w; ++c) {
        fixed[(size_t)o * w + c] = 0;
        if (!usable) continue;
        int64_t A = 0, B = kFxB0, C = kFxC0;
        for (int j = 0; j <= 2 * H; ++j) {
          const Fx f = fx_split(ring[(size_t)((o - H + j) % NR) * w + c]);
          A = fx_mad(t.w1[j], f.hi, A);
          B = fx_mad(t.w1[j], f.lo, B);
          C = fx_mad(t.w0[j], f.hi, C);
        }
        if (fx_upper((int32_t)(ring[(size_t)(o % NR) * w + c] >> 32)) < fx_least(10, lift)) continue;
        out[(size_t)o * w + c] = fx_to(fx_join(A, B, C), scale.E - 1023 - t.sw);
        fixed[(size_t)o * w + c] = 1;
      }
    }
    if (i >= np) continue;
    int mag = 0;
    for (int c = 0; c < w; ++c) {
      const int m = fx_mag(v[(size_t)i * w + c]);
      if (m > mag) mag = m;
      if (mag == 0 && fx_word(v[(size_t)i * w + c], 0) != 0) mag = 1;
    }
    const bool ok = fx_plane_usable(mag);
    const int top = ok ? mag >> 20 : 0, d = fx_ring_join(scale, planes, i, top, H, ok);
    fx_ring_note(planes, scale, i, top, d, ok);
    if (d != 0) for (auto &x : ring) x = fx_rescale(x, d);
    if (ok) for (int c = 0; c < w; ++c) ring[(size_t)(i % NR) * w + c] = fx_from(v[(size_t)i * w + c], scale.E);
  }
  return 1;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    src = d / "ring.cpp"
    src.write_text(SRC)
    so = str(d / "ring.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", ROOT, str(src), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


TAPS = {1: [0.05, 0.9, 0.05], 2: [-0.004, 0.07, 0.868, 0.07, -0.004], 3: [0.0005, -0.007, 0.07, 0.873, 0.07, -0.007, 0.0005]}


def _planes(kind, size, np_, w, rng):
    v = rng.uniform(0.5, 1.0, (np_, w)) * rng.choice([1.0, -1.0], (np_, w))
    if kind == "slab":
        v[9:11] *= size
    elif kind == "two_slabs":  # the second falls while planes cut under the first are still read
        v[9] *= size
        v[12] *= size ** 0.5
        v[25:] /= size
    elif kind == "decay":
        v *= (size ** -0.25) ** np.arange(np_)[:, None]
    elif kind == "rise":
        v *= (size ** 0.25) ** np.arange(np_)[:, None]
    elif kind == "unusable":  # planes with an infinity, a NaN, or values at the end of the exponent range
        v[7, 3], v[16, 5], v[28] = np.inf, np.nan, v[28] * 1e-280
        v[20:] /= size
        v[33] *= 1e-310 / np.abs(v[33]).max()
    elif kind == "waves":  # smooth along z, a few planes per sign change
        v = np.abs(v) * np.sin(0.5 * np.arange(np_) + 0.3)[:, None]
    return v


@pytest.mark.parametrize("H", [1, 2, 3])
@pytest.mark.parametrize("size", [4.0, 16.0, 1e4, 1e8, 1e12, 1e16, 1e20])
@pytest.mark.parametrize("kind", ["slab", "two_slabs", "decay", "rise", "unusable", "waves"])
def test_what_the_ring_lets_through_is_as_exact_as_a_chain(lib, kind, size, H):
    rng = np.random.default_rng([len(kind), H, int(np.log2(size))])
    np_, w, n = 40, 24, 2 * H + 1
    v = np.ascontiguousarray(_planes(kind, size, np_, w, rng))
    out, fixed = np.zeros((np_, w)), np.zeros((np_, w), dtype=np.uint8)
    P = ctypes.c_void_p
    assert lib.march(np_, w, v.ctypes.data_as(P), H, np.array(TAPS[H]).ctypes.data_as(P), out.ctypes.data_as(P),
                     fixed.ctypes.data_as(P))
    for o in range(H, np_ - H):
        for c in range(w):
            if not fixed[o, c]:
                continue
            assert kind != "unusable" or not {7, 16, 28, 33} & set(range(o - H, o + H + 1))
            terms = [Fraction(a) * Fraction(float(b)) for a, b in zip(TAPS[H], v[o - H:o + H + 1, c])]
            bound = Fraction(float(np.abs(v[o - H:o + H + 1, c]).max())) * (7 + n) * Fraction(1, 2 ** 53)
            assert abs(Fraction(float(out[o, c])) - sum(terms)) <= bound, (o, c)
    if kind == "waves":  # a smooth field stays in fixed point
        assert fixed[H:np_ - H].mean() > 0.9
