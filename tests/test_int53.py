"""Reciprocal and roots on integer significands (csrc/mhd_int53.cuh), on the
CPU: for any float seed inside the special-function unit's error bound the
reciprocal and the square root are the IEEE-rounded values, and the
reciprocal square root is within 0.51 ulp."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_05240_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include "mhd_int53.cuh"
using namespace mhd;
int main(int argc, char** argv) {
  const int kind = atoi(argv[1]);
  std::mt19937_64 g(17 + kind);
  const uint64_t all = (1ull << 52) - 1;
  long bad_rcp = 0, bad_sqrt = 0, bad_rsqrt = 0;
  for (long it = 0; it < 300000; ++it) {
    uint64_t f = g() & all;
    if (kind == 1) f &= 0xff;                // just above a power of two
    if (kind == 2) f = all - (g() & 0xff);   // just below one
    if (kind == 3) f = (f >> 26) << 26;      // short significands (exact squares, ties)
    if (kind == 4) f = it & 1 ? 0 : all;
    const uint64_t M = (1ull << 52) | f;
    const double x = (double)M * 0x1p-52;
    const float xf = (float)((double)(M >> 29) * 0x1p-23);
    for (int s = -2; s <= 2; ++s) {
      auto off = [&](double v) {
        float r = (float)v;
        for (int k = 0; k < std::abs(s); ++k) r = nextafterf(r, s > 0 ? 4.0f : 0.0f);
        return r;
      };
      bad_rcp += (double)rcp_sig(M, off(1.0 / xf)) * 0x1p-53 != 1.0 / x;
      for (int odd = 0; odd < 2; ++odd) {
        const double m = odd ? 2 * x : x;
        const float seed = off(1.0 / std::sqrt((double)xf * (odd ? 2 : 1)));
        bad_sqrt += (double)sqrt_sig(M, odd, seed) * 0x1p-52 != std::sqrt(m);
        const long double d = (long double)rsqrt_sig(M, odd, seed) - 0x1p53L / sqrtl((long double)m);
        bad_rsqrt += !(d < 0.51L && d > -0.51L);
      }
    }
  }
  printf("%ld %ld %ld\n", bad_rcp, bad_sqrt, bad_rsqrt);
  return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("int53")
    src, exe = d / "t.cpp", d / "t"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("kind", range(5))
def test_rounding_for_every_seed_in_the_bound(harness, kind):
    out = subprocess.run([harness, str(kind)], check=True, capture_output=True, text=True).stdout.split()
    assert [int(v) for v in out] == [0, 0, 0]


PRODUCTS = r"""
#include <cstdio>
#include <random>
#include "mhd_int53.cuh"
using namespace mhd;
int main() {
  std::mt19937_64 g(5);
  const uint64_t all = (1ull << 52) - 1;
  long bad = 0;
  for (long it = 0; it < 4000000; ++it) {
    uint64_t fa = g() & all, fb = g() & all;
    if (it % 8 == 1) fa &= 0xffff;                                    // 1 + ulps
    if (it % 8 == 2) fa = (fa >> 26) << 26, fb = (fb >> 26) << 26;      // exact products
    if (it % 8 == 3) fa = (fa >> 30) << 30, fb = (fb >> 20) << 20;      // ties
    if (it % 8 == 4) fa |= all ^ 0xff, fb |= all ^ 0xff;                // carries out of the significand
    if (it % 8 == 5) fa = 0;
    const uint64_t a = (1ull << 52) | fa, b = (1ull << 52) | fb;
    int big;
    const uint64_t q = mul_sig(a, b, big);
    bad += (double)q * 0x1p-52 * (big ? 2 : 1) != ((double)a * 0x1p-52) * ((double)b * 0x1p-52);
  }
  printf("%ld\n", bad);
  return 0;
}
"""


def test_products_are_ieee(tmp_path):
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PRODUCTS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip() == "0"
