"""The fixed-point complex logarithm and exponential of the FP64 kernels
(csrc/hpt_fx.cuh), compiled for the host: against long double.

Bounds: the header states about 2^-59 for log2|y|, 2^-60 revolution for the
angle and 2^-57.5 for the fractions of exp2 and sincos; the tests allow twice
that plus the rounding of the long double reference.  One monomial
(c y^a t^e, through log, sum and exp) is then a correctly rounded double up to
5%: 0.53 ulp of the modulus, 1.2e-16 per component.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include <math.h>
#include "hpt_fx.cuh"
using namespace hpt::fx;
typedef long double L;
static const L kPi = acosl(-1.0L);
static L mod16(L d) { return d - 16 * rintl(d / 16); }
extern "C" int log_err(long n, const double* re, const double* im, double* el, double* et, double* ef) {
  int bad = 0;
  for (long i = 0; i < n; ++i) {
    Log o;
    if (!log_of(re[i], im[i], o)) { ++bad; el[i] = et[i] = ef[i] = 0; continue; }
    const L l = log2l(hypotl((L)re[i], (L)im[i])), t = atan2l((L)im[i], (L)re[i]) / (2 * kPi);
    el[i] = (double)mod16((L)o.l / (L)(1ll << 60) - l);
    L d = ldexpl((L)(int64_t)o.turn, -64) - t;
    et[i] = (double)(d - rintl(d));
    ef[i] = (double)(o.lf - l);
  }
  return bad;
}
extern "C" void mono_err(long n, int nnz, const double* y, const int* a, const double* c, const int* e,
                         const double* tau, double* err) {
  for (long i = 0; i < n; ++i) {
    Log lg;
    log_of(c[2 * i], c[2 * i + 1], lg);
    const Wide w = log2e_times(tau[i]);
    int64_t W = lg.l + times(e[i], w);
    uint64_t th = lg.turn;
    float wf = lg.lf + (float)e[i] * ((float)tau[i] * 1.44269504f);
    L re = logl(hypotl((L)c[2 * i], (L)c[2 * i + 1])) + (L)e[i] * tau[i], im = atan2l((L)c[2 * i + 1], (L)c[2 * i]);
    for (int j = 0; j < nnz; ++j) {
      const double* v = y + 2 * (i * nnz + j);
      const int64_t k = a[i * nnz + j];
      log_of(v[0], v[1], lg);
      W += k * lg.l;
      th += (uint64_t)k * lg.turn;
      wf += (float)k * lg.lf;
      re += k * logl(hypotl((L)v[0], (L)v[1]));
      im += k * atan2l((L)v[1], (L)v[0]);
    }
    double er, ei;
    exp_of(W, th, wf, h_tables.exp1, h_tables.exp2, h_tables.cs1, h_tables.cs2, er, ei);
    const L m = expl(re);
    err[i] = (double)(hypotl(er - m * cosl(im), ei - m * sinl(im)) / m);
  }
}
extern "C" double exp_edge(double w) {
  const int64_t W = (int64_t)((w - 16 * rint(w / 16)) * (double)(1ll << 60));
  double er, ei;
  exp_of(W, 0, (float)w, h_tables.exp1, h_tables.exp2, h_tables.cs1, h_tables.cs2, er, ei);
  return er;
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    src = d / "fx.cpp"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2111_14317_gb300", "csrc"), str(src), "-o", str(d / "fx.so")], check=True)
    lib = ctypes.CDLL(str(d / "fx.so"))
    lib.exp_edge.restype = ctypes.c_double
    lib.exp_edge.argtypes = [ctypes.c_double]
    return lib


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


@pytest.mark.parametrize("spread", [0.0, 2.0, 60.0, 300.0, 1000.0])
def test_log(lib, spread):
    """Points of every octant, both axes, the diagonals, components up to 70
    binades apart, moduli over the double range (subnormals included)."""
    rng = np.random.default_rng(int(spread) + 1)
    n = 200_000
    s = np.exp2(np.floor(rng.uniform(-spread, min(spread, 1000.0), n)))
    re, im = rng.standard_normal(n) * s, rng.standard_normal(n) * s
    im[::7] *= np.exp2(-np.floor(rng.uniform(0, 70, len(im[::7]))))
    re[1::11] *= np.exp2(-np.floor(rng.uniform(0, 70, len(re[1::11]))))
    im[::1001] = 0.0
    re[1::1003] = 0.0
    re[2::1009] = im[2::1009]
    re[3::1013] = -im[3::1013]
    if spread == 1000.0:
        re[4::17] *= 1e-300
        im[4::17] *= 1e-300
    keep = (re != 0) | (im != 0)
    re, im = np.ascontiguousarray(re[keep]), np.ascontiguousarray(im[keep])
    el, et, ef = (np.empty(len(re)) for _ in range(3))
    assert lib.log_err(ctypes.c_long(len(re)), _p(re), _p(im), _p(el), _p(et), _p(ef)) == 0
    # the reference itself: long double has 64 bits here or more, log2 up to 1075
    assert np.abs(el).max() <= 2.0 ** -58 + 2.0 ** -63 * max(1.0, 2 * spread + 80)
    assert np.abs(et).max() <= 2.0 ** -59
    assert np.abs(ef).max() <= 1e-4


def test_log_refuses(lib):
    re = np.array([0.0, -0.0, np.inf, np.nan, 1.0, 1.0])
    im = np.array([0.0, 0.0, 1.0, 1.0, -np.inf, np.nan])
    out = [np.empty(6) for _ in range(3)]
    assert lib.log_err(ctypes.c_long(6), _p(re), _p(im), *[_p(o) for o in out]) == 6


@pytest.mark.parametrize("nnz,amax,emax", [(1, 2, 16), (4, 3, 64), (24, 2, 1 << 20), (3, 300, 1 << 30)])
def test_monomial(lib, nnz, amax, emax):
    rng = np.random.default_rng(nnz)
    n = 50_000
    y = np.exp(0.5 / max(1, amax / 8) * rng.standard_normal((n, nnz)) + 2j * np.pi * rng.random((n, nnz)))
    a = rng.integers(-amax, amax + 1, size=(n, nnz)).astype(np.int32)
    c = np.exp(rng.standard_normal(n) + 2j * np.pi * rng.random(n))
    e = rng.integers(0, emax + 1, size=n).astype(np.int32)
    tau = -rng.uniform(0, 20, n) / np.maximum(e, 1)
    err = np.empty(n)
    lib.mono_err(ctypes.c_long(n), nnz, _p(np.ascontiguousarray(y).view(np.float64)), _p(a), _p(c.view(np.float64)),
                 _p(e), _p(tau), _p(err))
    # sum |a| times the logarithms' errors (2^-59 ln 2 and 2^-60 2 pi) on top of the rounding to double
    assert err.max() <= 1.3e-16 + nnz * amax * (np.log(2) * 2.0 ** -59 + 2 * np.pi * 2.0 ** -60)


def test_exp_range(lib):
    """The ends of the double range: subnormals, zero, infinity."""
    for w in (-1000.5, -1022.0, -1030.25, 0.0, 1000.5, 1019.5, 1022.75):
        assert abs(lib.exp_edge(w) / 2.0 ** w - 1) < (1e-12 if w > -1021 else 2e-13 + 2.0 ** (-1074 - w))
    assert lib.exp_edge(-1080.0) == 0.0 and lib.exp_edge(-5000.0) == 0.0
    assert lib.exp_edge(1025.0) == np.inf
    assert np.isnan(lib.exp_edge(2000.0))
