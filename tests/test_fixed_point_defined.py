"""The fixed-point arithmetic of csrc/hpt_fx.cuh without undefined behaviour: a
host build that traps on signed overflow, bad shifts and bad conversions runs
the logarithm, exponent sums that wrap modulo 16 many times, and both
exponentials; and the kernels form their sums by the same functions."""
import os
import re
import subprocess

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2111_14317_gb300", "csrc")
SRC = r'''
#include <math.h>
#include <stdio.h>
#include "hpt_fx.cuh"
using namespace hpt::fx;
typedef long double L;
int main() {
  uint64_t x = 88172645463325252ull;
  auto rnd = [&x] { x ^= x << 13; x ^= x >> 7; x ^= x << 17; return x; };
  double worst = 0;
  for (int i = 0; i < 300000; ++i) {
    Sum s{0, 0, 0.f};
    const double tau = -(double)(rnd() % 1000) / 100;
    const int e = (int)(rnd() % 7);
    s.w += times(e, log2e_times(tau));
    s.f = (float)e * (float)tau * 1.44269504f;
    L re = (L)e * tau, im = 0;
    for (int j = 0; j < 8; ++j) {
      const int spread = i % 3 == 0 ? 30 : 2, a = (int)(rnd() % 41) - 20;
      const double m = ldexp(1.0 + (double)(rnd() >> 12) * 0x1p-52, (int)(rnd() % (2 * spread + 1)) - spread);
      const double ph = (double)(rnd() >> 11) * 0x1p-53 * 6.283185307179586;
      const double r = m * cos(ph), q = m * sin(ph);
      Log lg;
      if (!log_of(r, q, lg)) return 1;
      add_power(s, a, (uint64_t)lg.l, lg.turn, lg.lf);
      re += a * logl(hypotl(r, q));
      im += a * atan2l(q, r);
    }
    double er, ei;
    exp_of((int64_t)s.w, s.turn, s.f, h_tables.exp1, h_tables.exp2, h_tables.cs1, h_tables.cs2, er, ei);
    if (exp_in_range(s.f)) {
      double fr, fi;
      exp_in((int64_t)s.w, s.turn, s.f, h_tables.exp1, h_tables.exp2, h_tables.cs1, h_tables.cs2, fr, fi);
      if (fr != er || fi != ei) return 2;
      const L m = expl(re);
      const double err = (double)(hypotl(er - m * cosl(im), ei - m * sinl(im)) / m);
      worst = err > worst ? err : worst;
    }
  }
  printf("%.3e\n", worst);
  return 0;
}
'''


def test_no_undefined_behaviour(tmp_path):
    (tmp_path / "fx.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-fsanitize=undefined", "-fsanitize-undefined-trap-on-error", "-I", CSRC,
                    str(tmp_path / "fx.cpp"), "-o", str(tmp_path / "fx")], check=True)
    r = subprocess.run([str(tmp_path / "fx")], capture_output=True, text=True)
    assert r.returncode == 0, r.returncode
    # the bound of tests/test_fixed_point.py for 8 factors of up to 20
    assert float(r.stdout) <= 1.3e-16 + 8 * 20 * (np.log(2) * 2.0 ** -59 + 2 * np.pi * 2.0 ** -60)


def test_the_kernels_use_the_unsigned_sum():
    for f in ("hpt_eval64.cu", "hpt_solve.cu"):
        src = open(os.path.join(CSRC, f)).read()
        assert "fx::add_power(" in src
        assert not re.search(r"\(int64_t\)\s*[\w.]+\s*\*\s*\(int64_t\)\s*z\.", src)
