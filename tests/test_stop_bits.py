"""The CG loops' scalar tests on bit patterns against the floating-point tests
they stand for (CPU: common.cuh compiled for the host).

Every test is compared for zeros, subnormal and normal values, infinities and
NaNs of both signs; the stop test also at the values around its threshold,
where the exact measure ||r|| / ||b|| <= eps decides.  A stop test never
passes for a NaN, whatever its sign."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_08059_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>
#include "common.cuh"
using namespace mpcg;

static double from(unsigned long long b) { double v; memcpy(&v, &b, 8); return v; }
static int bad = 0;
static void check(bool ok, const char* what, double v, double w = 0.0) {
  if (!ok && ++bad <= 20) printf("%s: %a (%a)\n", what, v, w);
}

int main() {
  std::vector<double> vs = {0.0, from(1), 4.9e-310, 2.3e-308, 1e-290, 1e-200, 1e-20, 1e-10, 0.5, 1.0, 3.0, 1e10,
                            1e200, 1e290, 1.7e308, INFINITY, from(0x7ff0000000000001ull), from(0x7ff8000000000000ull),
                            from(0x7fffffffffffffffull)};
  unsigned long long s = 88172645463325252ull;
  for (int i = 0; i < 20000; ++i) {
    s ^= s << 13; s ^= s >> 7; s ^= s << 17;
    vs.push_back(from(s & 0x7fffffffffffffffull));
  }
  for (double a : vs)
    for (double v : {a, -a}) {
      check(bits_finite(v) == (bool)std::isfinite(v), "finite", v);
      check(bits_nan(v) == (bool)std::isnan(v), "nan", v);
      check(bits_positive(v) == (v > 0.0), "positive", v);
    }
  for (int rel : {0, 1})
    for (double bn : {1e-160, 1e-3, 1.0, 7.3, 1e6, 1e150})
      for (double eps : {0.0, 1e-300, 1e-15, 1e-10, 1e-4, 1.0, 1e3}) {
        const StopThr T = stop_thr(eps, bn, rel);
        std::vector<double> rr = vs;
        const double e = rel ? eps * bn : eps;
        for (double f : {1.0 - 1e-9, 1.0 - 1e-12, 1.0, 1.0 + 1e-12, 1.0 + 1e-9}) {
          double lo = e * e * f, hi = lo;
          for (int k = 0; k < 200; ++k) {
            rr.push_back(lo);
            rr.push_back(hi);
            lo = std::nextafter(lo, 0.0);
            hi = std::nextafter(hi, INFINITY);
          }
        }
        for (double v : rr) {
          check(stop_pass(T, v) == (stop_measure(v, bn, rel) <= eps), "stop", v, eps);
          if (std::isnan(v)) {
            check(!stop_pass(T, v), "stop on NaN", v, eps);
            check(!stop_pass(T, std::copysign(v, -1.0)), "stop on NaN with the sign bit", std::copysign(v, -1.0), eps);
          }
        }
      }
  printf("%d\n", bad);
  return bad != 0;
}
"""


def test_bit_tests_are_the_floating_point_tests(tmp_path):
    src, exe = tmp_path / "bits.cu", tmp_path / "bits"
    src.write_text(PROGRAM)
    r = subprocess.run([os.environ.get("NVCC", "nvcc"), "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-I", CSRC, "-o", str(exe), str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
