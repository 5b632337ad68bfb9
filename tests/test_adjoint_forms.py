"""Reverse of the forms that the stage kernels evaluate (interface_flux2_rev, source_pressure_rev,
smooth_rev) against the tangents of their forward functions on dual numbers: the dot products <ob, T u>
and <T^T ob, u> agree to 1e-12 of the sum of their terms' magnitudes. cell_rev_general, which passes the
adjoints of recon_cell_rev (pinned in test_adjoint_cells.py) on to fewer differences, against those
adjoints mapped to the averages directly."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2208_06588_gb300", "csrc")

FWD = r"""
#include <cmath>
#include <cstdint>
@DUAL@
#define SWALE_REAL dt::D
#include "swale_cell.cuh"
using dt::D;
using namespace swale;
static D q(const double* v, const double* d, int k) { return D(v[k], d[k]); }
extern "C" {
// e[8]: EL ER BL BR uL uR (hL, hR unused by the flux of this scheme); f[4]: FE FMl FMr FB
void t_flux(const double* prm, const double* e, const double* de, double* df) {
  Flux2 f = interface_flux2<0>(D(prm[0]), D(prm[1]), D(prm[2]), q(e, de, 0), q(e, de, 1), q(e, de, 2), q(e, de, 3), D(0.0),
                               D(0.0), q(e, de, 4), q(e, de, 5));
  df[0] = f.FE.d; df[1] = f.FMl.d; df[2] = f.FMr.d; df[3] = f.FB.d;
}
double t_source(const double* m, const double* a, const double* da) {
  SourceRatio s{D(m[4]), D(m[5]), D(m[6])};
  return source_pressure_form(q(a, da, 0), q(a, da, 1), q(a, da, 2), q(a, da, 3), q(a, da, 4), q(a, da, 5), q(a, da, 6),
                              q(a, da, 7), q(a, da, 8), D(m[0]), D(m[1]), D(m[2]), D(m[3]), s).d;
}
// One cell through differences, edge values and limiter, as the kernels do it: u[15] = averages of eta, hu, h
// on the five cells; out[8] the edge state's tangents; returns the class (-1: the limiter acted).
int t_cell(const double* h, const double* prm, const double* u, const double* du, double* out) {
  SchemeConst P{prm[0], prm[1], prm[2], prm[3], 1, (int32_t)prm[5]};
  D H[5], p[4], v[3], d2[3][4], d3[3][3], d4[3][2], ev[3][2];
  for (int k = 0; k < 5; ++k) H[k] = D(h[k]);
  for (int a = 0; a < 4; ++a) p[a] = H[a] + H[a + 1];
  for (int k = 0; k < 3; ++k) {
    v[k] = q(u, du, 5 * k + 2);
    for (int a = 0; a < 4; ++a) d2[k][a] = (q(u, du, 5 * k + a + 1) - q(u, du, 5 * k + a)) / p[a];
    for (int a = 0; a < 3; ++a) d3[k][a] = (d2[k][a + 1] - d2[k][a]) / (p[a] + H[a + 2]);
    for (int a = 0; a < 2; ++a) d4[k][a] = (d3[k][a + 1] - d3[k][a]) / (p[a] + p[a + 2]);
  }
  const D iv = D(1.0) / (p[0] + p[2] + H[4]);
  int cls = 0;
  for (int e = 0; e < 2; ++e) {
    D o[3];
    cls = open_edge_values(P, H, p, D(prm[4]), iv, v, d2, d3, d4, e == 1, o);
    for (int k = 0; k < 3; ++k) ev[k][e] = o[k];
  }
  EdgeState o;
  uint32_t st = 0;
  limit_cell(P, ev, v[2], v[1], o, st);
  const D r[8] = {o.EL, o.ER, o.BL, o.BR, o.hL, o.hR, o.uL, o.uR};
  for (int k = 0; k < 8; ++k) out[k] = r[k].d;
  return (o.hL.v != ev[2][0].v || o.hR.v != ev[2][1].v) ? -1 : cls;
}
}
"""

REV = r"""
#include <cmath>
#include <cstdint>
#include "swale_adjoint.cuh"
using namespace swale;
extern "C" {
void r_flux(const double* prm, const double* e, const double* fb, double* eb) {
  FaceAdj a = interface_flux2_rev(prm[0], prm[1], prm[2], e[0], e[1], e[2], e[3], e[4], e[5], fb[0], fb[1], fb[2], fb[3]);
  eb[0] = a.EL; eb[1] = a.ER; eb[2] = a.BL; eb[3] = a.BR; eb[4] = a.uL; eb[5] = a.uR;
}
void r_source(const double* m, const double* a, double ab, double* b) {
  SourceRatio s{m[4], m[5], m[6]};
  SourceAdj r = source_pressure_rev(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], m[0], m[1], m[2], m[3], s, ab);
  const double o[9] = {r.hc, r.hL, r.hR, r.deL, r.deR, r.dEl, r.dHl, r.dEr, r.dHr};
  for (int k = 0; k < 9; ++k) b[k] = o[k];
}
// mode 0: cell_rev_general; 1: smooth_rev with the limiter not active. ub[15]: adjoints of the averages.
void r_cell(const double* h, const double* prm, const double* u, const double* o, const double* ob, int mode, double* ub) {
  SchemeConst P{prm[0], prm[1], prm[2], prm[3], 1, (int32_t)prm[5]};
  EdgeAdj a{ob[0], ob[1], ob[2], ob[3], ob[4], ob[5], ob[6], ob[7]};
  SmoothAdj r[3];
  double p[4];
  for (int k = 0; k < 4; ++k) p[k] = h[k] + h[k + 1];
  if (mode == 0) {
    cell_rev_general(P, h, u, u + 5, u + 10, prm[4], a, r);
  } else {
    const SmoothWidths w = {h[1], h[2], h[3], p[0], p[1], p[2], p[3]};
    const double iv = 1.0 / (p[0] + p[2] + h[4]), mL = a.uL / o[4], mR = a.uR / o[5];
    r[0] = smooth_rev(w, iv, a.EL + a.BL, a.ER + a.BR);
    r[1] = smooth_rev(w, iv, mL, mR);
    r[2] = smooth_rev(w, iv, (a.hL - a.BL) - mL * o[6], (a.hR - a.BR) - mR * o[7]);
  }
  // the kernels' transpose of the differences, for one cell
  for (int v = 0; v < 3; ++v) {
    double d3[3] = {0, r[v].d3, 0}, d2[4] = {0, r[v].d2l, r[v].d2r, 0}, c[5] = {0, 0, r[v].v, 0, 0};
    const double d4[2] = {r[v].d4l, r[v].d4r};
    for (int a2 = 0; a2 < 2; ++a2) {
      const double t = d4[a2] / (p[a2] + p[a2 + 2]);
      d3[a2 + 1] += t;
      d3[a2] -= t;
    }
    for (int a2 = 0; a2 < 3; ++a2) {
      const double t = d3[a2] / (p[a2] + h[a2 + 2]);
      d2[a2 + 1] += t;
      d2[a2] -= t;
    }
    for (int a2 = 0; a2 < 4; ++a2) {
      const double t = d2[a2] / p[a2];
      c[a2 + 1] += t;
      c[a2] -= t;
    }
    for (int k = 0; k < 5; ++k) ub[5 * v + k] = c[k];
  }
}
// The same from recon_cell_rev's own adjoints (variables eta, hu, b), every difference transposed.
void r_plain(const double* h, const double* prm, const double* u, const double* ob, double* ub) {
  SchemeConst P{prm[0], prm[1], prm[2], prm[3], 1, (int32_t)prm[5]};
  EdgeAdj a{ob[0], ob[1], ob[2], ob[3], ob[4], ob[5], ob[6], ob[7]};
  double V[3][5], v0[3][3], v0b[3][3], it[3];
  StencilDD DD, DDb;
  for (int k = 0; k < 5; ++k) {
    V[0][k] = u[k];
    V[1][k] = u[5 + k];
    V[2][k] = u[k] - u[10 + k];
  }
  for (int q = 0; q < 3; ++q) it[q] = 1.0 / (h[q] + h[q + 1] + h[q + 2]);
  for (int v = 0; v < 3; ++v) {
    for (int k = 0; k < 3; ++k) v0[v][k] = V[v][k];
    for (int k = 0; k < 4; ++k) DD.D2[v][k] = (V[v][k + 1] - V[v][k]) * (1.0 / (h[k] + h[k + 1]));
    for (int k = 0; k < 3; ++k) DD.D3[v][k] = (DD.D2[v][k + 1] - DD.D2[v][k]) * it[k];
  }
  recon_cell_rev(P, h, it, v0, DD, prm[4], a, v0b, DDb, false);
  for (int v = 0; v < 3; ++v) {
    double d2[4], c[5] = {v0b[v][0], v0b[v][1], v0b[v][2], 0, 0};
    for (int k = 0; k < 4; ++k) d2[k] = DDb.D2[v][k];
    for (int k = 0; k < 3; ++k) {
      const double t = DDb.D3[v][k] * it[k];
      d2[k + 1] += t;
      d2[k] -= t;
    }
    for (int k = 0; k < 4; ++k) {
      const double t = d2[k] / (h[k] + h[k + 1]);
      c[k + 1] += t;
      c[k] -= t;
    }
    for (int k = 0; k < 5; ++k) ub[5 * v + k] = c[k];
  }
  for (int k = 0; k < 5; ++k) {  // b = eta - h
    ub[k] += ub[10 + k];
    ub[10 + k] = -ub[10 + k];
  }
}
}
"""


@pytest.fixture(scope="module")
def libs(tmp_path_factory):
    d = tmp_path_factory.mktemp("adjforms")
    dual = open(os.path.join(ROOT, "tests", "cellcheck", "celltest_tangent.cpp")).read()
    dual = re.search(r"namespace dt \{.*?\}  // namespace dt", dual, re.S).group(0)
    out = []
    for name, src in (("fwd", FWD.replace("@DUAL@", dual)), ("rev", REV)):
        f, so = d / f"{name}.cpp", d / f"{name}.so"
        f.write_text(src)
        subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, "-o", str(so), str(f)], check=True)
        out.append(ctypes.CDLL(str(so)))
    out[0].t_source.restype = ctypes.c_double
    out[0].t_cell.restype = ctypes.c_int
    return out


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _dots(a, b, c, d):
    """<a, b> against <c, d>, to 1e-12 of the magnitudes."""
    assert abs(a @ b - c @ d) <= 1e-12 * (np.abs(a) @ np.abs(b) + np.abs(c) @ np.abs(d))


def test_flux_and_source(libs):
    F, R = libs
    rng = np.random.default_rng(1)
    for _ in range(300):
        prm = np.array([9.812, 8.0, rng.uniform(-2, 2)])
        E, h, u = rng.uniform(0, 2, 2), rng.uniform(0, 2, 2), rng.uniform(-3, 3, 2)
        e = np.array([*E, *(E - h), *u])
        de, fb, df, eb = rng.normal(size=6), rng.normal(size=4), np.zeros(4), np.zeros(6)
        F.t_flux(_p(prm), _p(e), _p(de), _p(df))
        R.r_flux(_p(prm), _p(e), _p(fb), _p(eb))
        _dots(fb, df, eb, de)
        m, a, da, b = rng.uniform(-1, 1, 7), rng.uniform(-1, 2, 9), rng.normal(size=9), np.zeros(9)
        t = F.t_source(_p(m), _p(a), _p(da))
        ab = rng.normal()
        R.r_source(_p(m), _p(a), ctypes.c_double(ab), _p(b))
        _dots(np.array([ab]), np.array([t]), b, da)


@pytest.mark.parametrize("limit_hu", [0, 1])
def test_cell(libs, limit_hu):
    """Every class and the active limiter through cell_rev_general; the smooth class through it and through
    smooth_rev against the tangent."""
    F, R = libs
    rng = np.random.default_rng(2)
    seen = {-1: 0, 0: 0, 1: 0, 2: 0}
    for i in range(3000):
        h = 0.1 * np.exp(rng.uniform(-0.6, 0.6, 5))
        amp = 10.0 ** rng.uniform(-4, 0.3)
        base = rng.choice([1.0, 0.05])
        hh = np.maximum(1e-3, base + amp * rng.uniform(-1, 1, 5) * rng.choice([1.0, 0.3]))
        if i % 3 == 0:
            hh = base + amp * np.linspace(0, 1, 5) ** 2
        u = np.concatenate([hh + amp * rng.uniform(-1, 1, 5), rng.uniform(-1, 1) + amp * rng.uniform(-1, 1, 5), hh])
        prm = np.array([9.812, 1e-6, 1e-11, 1e-6, h.max(), limit_hu])
        du, ob, out, ub, val = rng.normal(size=15), rng.normal(size=8), np.zeros(8), np.zeros(15), np.zeros(8)
        cls = F.t_cell(_p(h), _p(prm), _p(u), _p(du), _p(out))
        seen[cls] += 1
        R.r_cell(_p(h), _p(prm), _p(u), _p(val), _p(ob), 0, _p(ub))
        ref = np.zeros(15)
        R.r_plain(_p(h), _p(prm), _p(u), _p(ob), _p(ref))
        # (the outer differences pass through sums of four widths: within a factor of 16 of the terms)
        assert np.abs(ub - ref).max() <= 16 * 1e-12 * max(1.0, np.abs(ref).max())
        if cls == 0:
            _dots(ob, out, ub, du)
            o = np.zeros(8)
            t = np.zeros(8)
            F.t_cell(_p(h), _p(prm), _p(u), _p(u), _p(t))  # linear in (eta, hu, h) but for u = m / h
            o[:6] = t[:6]
            z = u.copy()
            z[10:] = 0.0
            F.t_cell(_p(h), _p(prm), _p(u), _p(z), _p(t))  # tangent along (eta, hu, 0): u's is m / h
            o[6:] = t[6:]
            R.r_cell(_p(h), _p(prm), _p(u), _p(o), _p(ob), 1, _p(ub))
            _dots(ob, out, ub, du)
    assert all(v > 30 for v in seen.values()), seen
