"""The scalar arithmetic of the device headers, compiled for the host against
stand-ins of the CUDA builtins (tests/host_cuda): the double functions on the
integer pipes against the IEEE operations, signs, zeros, infinities, NaN and
every exponent at the ends of the range included."""
import os
import subprocess

import pytest

TESTS = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(TESTS), "paper_2402_05240_gb300", "csrc")

PRELUDE = r"""
#define MHD_HOST_CHECK 1
#include "cuda_runtime.h"
#include "mhd_adjoint.cuh"
#include <cstdio>
#include <cstdlib>
#include <limits>
#include <random>
#include <vector>
using namespace mhd;
static bool same(double a, double b) { return dbits(a) == dbits(b) || (a != a && b != b); }
// both signs of: zeros, infinities, NaN, and random, round and extreme
// significands at each end of the exponent range and in its middle
static std::vector<double> values(int per) {
  std::mt19937_64 g(11);
  std::vector<double> v = {0.0, std::numeric_limits<double>::infinity(), std::numeric_limits<double>::quiet_NaN()};
  const int ends[] = {0, 1, 2, 3, 4, 5, 480, 511, 512, 534, 535, 1021, 1022, 1023, 1024, 1533, 1534, 2040,
                      2041, 2042, 2043, 2044, 2045, 2046};
  const uint64_t all = (1ull << 52) - 1;
  for (int e : ends)
    for (int i = 0; i < per; ++i) {
      uint64_t f = i == 0 ? 0 : i == 1 ? all : i == 2 ? 1 : i == 3 ? all ^ 1 : i == 4 ? 3 : i == 5 ? 1ull << 51 : g() & all;
      v.push_back(word_cast<double>(((uint64_t)e << 52) | f));
    }
  const size_t n = v.size();
  for (size_t i = 0; i < n; ++i) v.push_back(-v[i]);
  return v;
}
"""


def compile_and_run(tmp_path, main, *args, flags=()):
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(PRELUDE + main)
    subprocess.run(["g++", "-O2", "-std=c++17", "-w", *flags, "-I", os.path.join(TESTS, "host_cuda"), "-I", CSRC,
                    str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe), *map(str, args)], check=True, capture_output=True, text=True).stdout.split()


INT_PIPE = r"""
int main() {
  const std::vector<double> v = values(40);
  long wrong = 0, unflagged = 0, flagged = 0;
  // a result in range is the IEEE one (the reciprocal root: within an ulp),
  // out of it the flag is set; the complete functions are right everywhere
  auto check = [&](bool bad, double got, double full, double ref, bool covered, double ulps) {
    auto off = [&](double x) { return ulps == 0 ? !same(x, ref) : !(same(x, ref) || fabs(x - ref) <= ulps * 0x1p-52 * ref); };
    if (!bad && off(got)) ++unflagged;
    if (bad && covered) ++flagged;
    if (off(full)) ++wrong;
  };
  auto normal = [](double x) { return fabs(x) >= 0x1p-1022 && fabs(x) <= 0x1.fffffffffffffp1023; };
  for (double x : v) {
    bool b = false;
    double r = rcp_try(x, b);
    check(b, r, rcp_int(x), 1.0 / x, normal(x) && normal(1.0 / x) && fabs(x) < 0x1p1022, 0);
    b = false;
    r = sqrt_try(x, b);
    check(b, r, sqrt_int(x), std::sqrt(x), x == 0 || (x > 0 && normal(x)), 0);
    b = false;
    r = rsqrt_try(x, b);
    check(b, r, rsqrt_int(x), (double)(1.0L / sqrtl((long double)x)), x > 0 && normal(x), 1.0);
  }
  for (double x : v)
    for (double y : v) {
      bool b = false;
      const double r = mul_try(x, y, b);
      check(b, r, mul_call(x, y), x * y, normal(x) && normal(y) && fabs(x * y) >= 0x1p-1021 && normal(2 * fabs(x) * y), 0);
    }
  printf("%ld %ld %ld\n", wrong, unflagged, flagged);
}
"""


def test_integer_pipe_functions(tmp_path):
    assert compile_and_run(tmp_path, INT_PIPE) == ["0", "0", "0"]
