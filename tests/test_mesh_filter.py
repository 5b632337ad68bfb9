"""The fixed-point sum of the fluid-driven mesh's filter (a g++ build of swale_cell.cuh) against integers of
any size: exact for every window that a configuration may ask for, up to 129 taps. Where it stands in for the
FP64 sum it is at least as accurate."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TOP_W = 1 << 56

SRC = r"""
#include "swale_cell.cuh"
using namespace swale;
extern "C" {
long long t_fixed(double v, int ex, int bits) { const Limbs l = fixed_point(v, ex, bits); return (long long)l.hi * (1ll << 28) + l.lo; }
long long t_sum(const long long* x, const long long* w, int n) {
  Limbs a[129], b[129];
  for (int i = 0; i < n; ++i) { a[i] = limbs(x[i]); b[i] = limbs(w[i]); }
  return filter_sum(a, b, n);
}
// One window: the FP64 sum and the fixed-point one (before the division by the weights' sum); returns whether the latter is
// taken.
int t_bits(int n) { return filter_bits(n); }
int t_window(const double* v, const double* w, int n, int ex, double* out) {
  Limbs a[129], b[129];
  double s = 0.0;
  for (int i = 0; i < n; ++i) {
    a[i] = fixed_point(v[i], ex, filter_bits(n));
    b[i] = limbs(llrint(ldexp(w[i], 56)));
    s = fma(w[i], v[i], s);
  }
  out[0] = s;
  out[1] = ldexp((double)filter_sum(a, b, n), ex - 1022 - filter_bits(n));
  return filter_fits(a, b, n / 2, filter_need(b, n));
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
    L.t_fixed.argtypes = [ctypes.c_double, ctypes.c_int, ctypes.c_int]
    return L


def exponent(v):
    """ex with |v| < 2^(ex - 1022): the biased exponent."""
    return int(np.abs(np.float64(v)).view(np.uint64) >> np.uint64(52))


@pytest.mark.parametrize("bits", [55, 56, 57, 58])
def test_fixed_point(lib, bits):
    rng = np.random.default_rng(1)
    for k in range(4000):
        top = np.ldexp(rng.uniform(1.0, 2.0), int(rng.integers(-300, 300)))
        v = rng.choice([-1, 1]) * top * 2.0 ** -rng.uniform(0, 70 if k % 2 else 3)
        ex = exponent(top)
        exact = Fraction(float(v)) * Fraction(2) ** (1022 + bits - ex)
        got = lib.t_fixed(v, ex, bits)
        assert abs(got) <= 1 << bits and abs(got - exact) <= Fraction(1, 2)
        if abs(v) >= 0.25 * 2.0 ** (ex - 1022):
            assert got == exact


@pytest.mark.parametrize("n", [1, 3, 31, 33, 49, 63, 65, 85, 97, 127, 129])
def test_sum_is_exact(lib, n):
    rng = np.random.default_rng(n)
    full, top = (1 << 28) - 1, 1 << lib.t_bits(n)
    xs = [np.full(n, v) for v in (top, -top, top - 1, 1 - top, full, -full, -1)]
    xs += [rng.integers(-top, top, n, endpoint=True) for _ in range(20)]
    ws = [np.full(n, v) for v in (TOP_W, TOP_W - 1, full, TOP_W - full)]
    ws += [np.rint(np.exp(-np.arange(-(n // 2), n // 2 + 1) ** 2 / (2 * s * s)) * 2.0 ** 56).astype(np.int64)
           for s in (0.3, 1.0, 8.0, 30.0, 64.0, 100.0, 400.0, 1e4)]
    for x in xs:
        for w in ws:
            x, w = np.ascontiguousarray(x, np.int64), np.ascontiguousarray(w, np.int64)
            got = lib.t_sum(x.ctypes.data_as(ctypes.c_void_p), w.ctypes.data_as(ctypes.c_void_p), n)
            exact = sum(int(a) * int(b) for a, b in zip(x, w))
            assert got == (exact + (1 << 55)) >> 56


@pytest.mark.parametrize("sigma", [0.3, 1.0, 8.0, 64.0, 1e4])
@pytest.mark.parametrize("half", [0, 1, 4, 24, 64])
def test_taken_where_it_is_as_accurate_as_fp64(lib, half, sigma):
    """Velocities of a tile (255 nodes and the window) of several kinds, every node's sum in both forms against the exact
    one. Where the fixed-point sum is taken its error is within its bound, (W + 1) 2^-56 + (2 H + 1) 2^-57 of the
    scale and the conversion's 2^-53 of the value, and over a tile its mean square is no larger than the FP64 sum's. It is
    not taken in quiet water."""
    n = 2 * half + 1
    w = np.exp(-np.arange(-half, half + 1.0) ** 2 / (2 * sigma * sigma))
    wf = [Fraction(float(a)) for a in w]
    rng = np.random.default_rng(half)
    m = 255 + 2 * half
    t = np.linspace(0.0, 1.0, m)
    fields = [1.0 + 0.3 * np.sin(7 * t), rng.uniform(-1, 1, m), np.sin(12 * t), np.where(t < 0.5, 1.7, 1e-9),
              np.exp(-30 * t), np.full(m, 1.99)]
    taken = 0
    for v in fields:
        ex = exponent(np.abs(v).max())
        unit = Fraction(2) ** (ex - 1022)
        sq = [Fraction(0), Fraction(0)]
        for i in range(0, 255, 7 if half < 64 else 31):
            win = np.ascontiguousarray(v[i:i + n])
            out = np.zeros(2)
            ok = lib.t_window(win.ctypes.data_as(ctypes.c_void_p), w.ctypes.data_as(ctypes.c_void_p), n, ex,
                              out.ctypes.data_as(ctypes.c_void_p))
            if np.abs(win).max() < 0.9 * 2.0 ** (ex - 1022 + 53 - lib.t_bits(n)):
                assert not ok
            if not ok:
                continue
            taken += 1
            exact = sum(a * Fraction(float(b)) for a, b in zip(wf, win))
            err = [abs(Fraction(float(o)) - exact) for o in out]
            bound = unit * ((sum(wf) + 1) / 2 ** 56 + Fraction(n, 2 ** 57)) + abs(exact) / 2 ** 53
            assert err[1] <= bound
            sq = [a + e * e for a, e in zip(sq, err)]
        assert sq[1] <= sq[0]
    assert taken > 0
