"""fast_div and fdiv of csrc/fastdiv.cuh, compiled for the host, against whole-number division: they give the PE and the group
of every 1D group of points."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "paper_1702_00496_gb300/csrc/fastdiv.cuh"
extern "C" int64_t wrong(uint32_t d, const uint32_t *n, int64_t count) {
  const atfd::FastDiv f = atfd::fast_div(d);
  int64_t bad = 0;
  for (int64_t i = 0; i < count; ++i) bad += atfd::fdiv(n[i], f) != n[i] / d;
  return bad;
}
"""
TOP = 2 ** 30


@pytest.fixture(scope="module")
def wrong(tmp_path_factory):
    d = tmp_path_factory.mktemp("div")
    src = d / "div.cpp"
    src.write_text(SRC)
    so = str(d / "div.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", ROOT, str(src), "-o", so], check=True)
    fn = ctypes.CDLL(so).wrong
    fn.restype = ctypes.c_int64
    fn.argtypes = [ctypes.c_uint32, ctypes.c_void_p, ctypes.c_int64]
    return lambda d, n: fn(d, n.ctypes.data, n.size)


def test_quotients_of_every_kind_of_divisor(wrong):
    rng = np.random.default_rng(3)
    near = [v for k in range(31) for v in (2 ** k - 1, 2 ** k, 2 ** k + 1)]
    divisors = [v for v in set(near + list(range(1, 300)) + [int(v) for v in rng.integers(1, TOP, 400)]) if 1 <= v < TOP]
    for d in divisors:
        q = rng.integers(0, (TOP - 1) // d + 1, 200)
        n = np.concatenate([q * d, q * d + d - 1, q * d - 1, rng.integers(0, TOP, 200), [0, 1, d - 1, d, d + 1, TOP - 1]])
        n = np.ascontiguousarray(n[(n >= 0) & (n < TOP)].astype(np.uint32))
        assert wrong(d, n) == 0, d


@pytest.mark.parametrize("d", [1, 2, 3, 62, 1022, 4097])
def test_every_numerator_of_a_large_grid(wrong, d):
    assert wrong(d, np.arange(1 << 22, dtype=np.uint32)) == 0
