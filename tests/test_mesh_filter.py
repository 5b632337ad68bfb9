"""The fixed-point sum of the fluid-driven mesh's filter (a g++ build of swale_cell.cuh) against integers of
any size: exact for every window that a configuration may ask for, up to 129 taps."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TOP_X, TOP_W = 1 << 55, 1 << 56

SRC = r"""
#include "swale_cell.cuh"
using namespace swale;
extern "C" {
long long t_fixed(double v, int ex) { const Limbs l = fixed_point(v, ex); return (long long)l.hi * (1ll << 28) + l.lo; }
long long t_sum(const long long* x, const long long* w, int n) {
  Limbs a[129], b[129];
  for (int i = 0; i < n; ++i) { a[i] = limbs(x[i]); b[i] = limbs(w[i]); }
  return filter_sum(a, b, n);
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("filter")
    src, so = d / "f.cpp", d / "f.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fsanitize=signed-integer-overflow,shift", "-fsanitize-undefined-trap-on-error",
                    "-I", os.path.join(ROOT, "paper_2208_06588_gb300", "csrc"), "-o", str(so),
                    str(src)], check=True)
    L = ctypes.CDLL(str(so))
    L.t_fixed.restype = L.t_sum.restype = ctypes.c_longlong
    L.t_fixed.argtypes = [ctypes.c_double, ctypes.c_int]
    return L


def exponent(v):
    """ex with |v| < 2^(ex - 1022): the biased exponent."""
    return int(np.abs(np.float64(v)).view(np.uint64) >> np.uint64(52))


def test_fixed_point(lib):
    rng = np.random.default_rng(1)
    for k in range(4000):
        top = np.ldexp(rng.uniform(1.0, 2.0), int(rng.integers(-300, 300)))
        v = rng.choice([-1, 1]) * top * 2.0 ** -rng.uniform(0, 70 if k % 2 else 3)
        ex = exponent(top)
        exact = Fraction(float(v)) * Fraction(2) ** (1022 + 55 - ex)
        got = lib.t_fixed(v, ex)
        assert abs(got) <= TOP_X and abs(got - exact) <= Fraction(1, 2)
        if abs(v) >= 0.25 * 2.0 ** (ex - 1022):
            assert got == exact


@pytest.mark.parametrize("n", [1, 3, 49, 63, 65, 85, 97, 127, 129])
def test_sum_is_exact(lib, n):
    rng = np.random.default_rng(n)
    full = (1 << 28) - 1
    xs = [np.full(n, v) for v in (TOP_X, -TOP_X, TOP_X - 1, 1 - TOP_X, full, -full, -1)]
    xs += [rng.integers(-TOP_X, TOP_X, n, endpoint=True) for _ in range(20)]
    ws = [np.full(n, v) for v in (TOP_W, TOP_W - 1, full, TOP_W - full)]
    ws += [np.rint(np.exp(-np.arange(-(n // 2), n // 2 + 1) ** 2 / (2 * s * s)) * 2.0 ** 56).astype(np.int64)
           for s in (0.3, 1.0, 8.0, 30.0, 64.0, 100.0, 400.0, 1e4)]
    for x in xs:
        for w in ws:
            x, w = np.ascontiguousarray(x, np.int64), np.ascontiguousarray(w, np.int64)
            got = lib.t_sum(x.ctypes.data_as(ctypes.c_void_p), w.ctypes.data_as(ctypes.c_void_p), n)
            exact = sum(int(a) * int(b) for a, b in zip(x, w))
            assert got == (exact + (1 << 55)) >> 56
