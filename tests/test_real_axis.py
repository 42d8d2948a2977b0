"""What is real stays real in FP64: phases that are whole quarter turns give
exactly 0 and +-1 (host build of csrc/hpt_fx.cuh), and real systems at real
points, their directions and start points on the axes come out without an
imaginary (or real) part (GPU)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "hpt_fx.cuh"
using namespace hpt::fx;
extern "C" void phase(uint64_t th, int64_t* c, int64_t* s) {
  cossin(th, h_tables.cs1, h_tables.cs2, *c, *s);
}
extern "C" void power(double re, double im, int a, double* er, double* ei) {
  Log lg;
  log_of(re, im, lg);
  exp_of((int64_t)((uint64_t)(int64_t)a * (uint64_t)lg.l), (uint64_t)(int64_t)a * lg.turn, (float)a * lg.lf, h_tables.exp1,
         h_tables.exp2, h_tables.cs1, h_tables.cs2, *er, *ei);
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2111_14317_gb300", "csrc"), str(d / "fx.cpp"), "-o", str(d / "fx.so")],
                   check=True)
    return ctypes.CDLL(str(d / "fx.so"))


def test_quarter_turns(lib):
    c, s = ctypes.c_int64(), ctypes.c_int64()
    one = 1 << 62
    for q, want in enumerate([(one, 0), (0, one), (-one, 0), (0, -one)]):
        lib.phase(ctypes.c_uint64(q << 62), ctypes.byref(c), ctypes.byref(s))
        assert (c.value, s.value) == want


@pytest.mark.parametrize("v", [1.0, 2.0, -3.0, 0.7, -1e-9, 2.5e40])
@pytest.mark.parametrize("a", [-3, -1, 1, 2, 7])
def test_powers_on_the_axes(lib, v, a):
    er, ei = ctypes.c_double(), ctypes.c_double()
    lib.power(ctypes.c_double(v), ctypes.c_double(0.0), a, ctypes.byref(er), ctypes.byref(ei))
    assert ei.value == 0.0 and abs(er.value / v ** a - 1) < 1e-15
    lib.power(ctypes.c_double(0.0), ctypes.c_double(v), a, ctypes.byref(er), ctypes.byref(ei))   # (i v)^a
    want = [(1, 0), (0, 1), (-1, 0), (0, -1)][a % 4]
    for got, unit in ((er.value, want[0]), (ei.value, want[1])):
        assert got == 0.0 if unit == 0 else abs(got / (unit * v ** a) - 1) < 1e-15


@pytest.mark.gpu
@pytest.mark.parametrize("proj", [False, True], ids=["affine", "projective"])
@pytest.mark.parametrize("n", [1, 5, 16, 19])
def test_real_system_at_real_points(hpt, n, proj):
    import torch

    s = W.laurent_system(3 + n, n, 3 if n == 1 else 6, -2, 2, 8, nnz=min(n, 3))
    rng = np.random.default_rng(n)
    s.coeffs[:] = rng.standard_normal(s.M)
    h = hpt.System.from_laurent(s, {"kind": "lower", "alpha_num": [0] * n, "denom": 1}, 0)
    if proj:
        h = h.homogenize()
    y = rng.uniform(0.5, 1.5, (70, h.nv)) * rng.choice([-1.0, 1.0], (70, h.nv))
    yd = torch.from_numpy(y).to(torch.complex128).cuda()
    t = torch.from_numpy(rng.uniform(0.2, 1.0, 70)).cuda()
    out = list(h.eval(yd, t))
    dE, dN, ok = h.euler_newton(yd, torch.log(t))
    assert ok.all()
    for a in out + [dE, dN]:
        assert (a.imag == 0).all() and (a.real != 0).any()


@pytest.mark.gpu
def test_start_points_on_the_axes(hpt):
    """Binomials with coefficients 1 and -1: every coordinate is a root of
    unity, and those that are +-1 or +-i are so exactly."""
    rng = np.random.default_rng(7)
    seen = 0
    for _ in range(40):
        n = int(rng.integers(2, 5))
        V = rng.integers(-4, 5, size=(n, n))
        if round(abs(np.linalg.det(V))) in (0, 1):
            continue
        exps = np.zeros((2 * n, n), np.int32)
        exps[1::2] = V
        y0, _ = hpt.binomial_start_device(n, [2] * n, exps, [-1, 1] * n, [[0, 1]] * n)
        y = y0.cpu().numpy()
        axis = np.round(y)
        near = np.abs(y - axis) < 1e-6
        near &= np.abs(axis) == 1
        assert (y[near] == axis[near]).all()
        seen += int(near.sum())
    assert seen > 200
