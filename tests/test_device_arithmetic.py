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


TINY_DIFFERENCES = r"""
// A cell with slopes of order one in density, normal velocity and pressure and
// differences of size d in its transverse components, which are of order 1e-37
// (a float pair made from a double below 2^-126 is zero; a difference of two
// may be any subnormal).
template <class T> static void cells(double d, T (*w)[7]) {
  const double x = d == 0.0 ? 0.0 : 1e-37 + 4 * d;
  const double base[7] = {1.0, 0.3, x, x, 0.8, x, x}, slope[7] = {0.2, -0.1, d, 1.5 * d, 0.15, 2.0 * d, -d};
  for (int m = 0; m < 3; ++m)
    for (int q = 0; q < 7; ++q) w[m][q] = T(base[q] + slope[q] * (m - 1) * (q < 2 || q == 4 ? 1.0 + 0.3 * (m - 1) : 1.0));
}
int main() {
  typedef TYPE T;
  long bad = 0;
  for (double d : {1e-45, 1e-42, 5e-40, 1e-39, 2.5e-39, 3.5e-39, 1e-38, 1e-37, 1e-30, 1e-24, 1e-19}) {
    T a[7], b[7], g[7];
    for (int q = 0; q < 7; ++q) {
      a[q] = T((float)(q & 1 ? d : -d));
      b[q] = T((float)(q & 1 ? 0.5 * d : -0.5 * d));
    }
    van_leer7<T>(a, b, g);  // the harmonic mean 2 d / 3, or 0 where a product underflows
    for (int q = 0; q < 7; ++q) {
      const double x = fabs(to_d<T>(g[q]));
      bad += !(x <= 1.01 * d + 1e-45);
    }
    T w[3][7], z[3][7], wl[7], wr[7], zl[7], zr[7];
    cells<T>(d, w);
    cells<T>(0.0, z);
    Ops<T> o;
    plmc<T>(o, T(5.0 / 3.0), w[0], w[1], w[2], T(0.4), wl, wr);
    plmc<T>(o, T(5.0 / 3.0), z[0], z[1], z[2], T(0.4), zl, zr);
    // differences of size d change the states by some d
    for (int q = 0; q < 7; ++q) {
      bad += !(fabs(to_d<T>(wl[q]) - to_d<T>(zl[q])) <= 1e-12 + 100 * d);
      bad += !(fabs(to_d<T>(wr[q]) - to_d<T>(zr[q])) <= 1e-12 + 100 * d);
    }
    T gl[7], gr[7], gm[7], g0[7], gp[7], gbn = T(0);
    for (int q = 0; q < 7; ++q) {
      gl[q] = T(1.0 - 0.1 * q);
      gr[q] = T(0.5 + 0.2 * q);
      gm[q] = g0[q] = gp[q] = T(0);
    }
    plmc_vjp<T>(T(5.0 / 3.0), T(1e-20), T(1e-20), w[0], w[1], w[2], T(0.4), gl, gr, gm, g0, gp, gbn);
    bad += !std::isfinite(to_d<T>(gbn));
    for (int q = 0; q < 7; ++q)
      bad += !std::isfinite(to_d<T>(gm[q])) + !std::isfinite(to_d<T>(g0[q])) + !std::isfinite(to_d<T>(gp[q]));
  }
  printf("%ld\n", bad);
}
"""


@pytest.mark.parametrize("typ", ["df", "double", "float"])
def test_plmc_with_tiny_differences(tmp_path, typ):
    """Differences whose product underflows leave van Leer's mean at zero."""
    assert compile_and_run(tmp_path, TINY_DIFFERENCES.replace("TYPE", typ)) == ["0"]


DOUBLING = r"""
int main() {
  long bad = 0;
  for (double x : values(60)) bad += !same(twice<double>(x), 2.0 * x);
  printf("%ld\n", bad);
}
"""


def test_doubling_is_the_ieee_one(tmp_path):
    assert compile_and_run(tmp_path, DOUBLING) == ["0"]


SCALINGS = r"""
int main() {
  long h = 0, qt = 0, qd = 0;
  for (double x : values(60)) {
    // (results below 2^-1022 are cut, not rounded: the largest would round to it)
    auto off = [](double r, double ref) { return fabs(ref) <= 0x1p-1022 ? !(fabs(r - ref) <= 0x1p-1074) : !same(r, ref); };
    h += off(half<double>(x), 0.5 * x);
    qt += off(quarter<double>(x), 0.25 * x);
    qd += !same(quad<double>(x), 4.0 * x);
  }
  printf("%ld %ld %ld\n", h, qt, qd);
}
"""


def test_scalings_at_the_ends_of_the_range(tmp_path):
    assert compile_and_run(tmp_path, SCALINGS) == ["0", "0", "0"]


NONFINITE = r"""
// outputs of a reverse function that respond to cotangent q have to be
// non-finite where that cotangent is
template <class F> static long lost(int nin, int nout, F f) {
  long bad = 0;
  std::vector<double> g(nin), o(nout), r(nout);
  for (int q = 0; q < nin; ++q)
    for (double x : {std::numeric_limits<double>::infinity(), std::numeric_limits<double>::quiet_NaN()}) {
      for (int k = 0; k < nin; ++k) g[k] = k == q ? 1.0 : 0.0;
      f(g.data(), o.data());
      for (int k = 0; k < nin; ++k) g[k] = k == q ? x : 0.1 + k;
      f(g.data(), r.data());
      for (int k = 0; k < nout; ++k) bad += o[k] != 0.0 && std::isfinite(r[k]);
    }
  return bad;
}
int main() {
  typedef TYPE T;
  std::mt19937_64 rng(5);
  std::normal_distribution<double> n;
  long hlld = 0, ppmc = 0, plmc = 0;
  for (int it = 0; it < 300; ++it) {
    double w[5][7], bn = n(rng);
    const double base[7] = {exp(0.3 * n(rng)), (it % 3) * n(rng), n(rng), n(rng), exp(0.3 * n(rng)), 0.5 * n(rng), 0.5 * n(rng)};
    double slope[7];
    for (double& s : slope) s = 0.05 * n(rng);
    for (int m = 0; m < 5; ++m)
      for (int q = 0; q < 7; ++q) w[m][q] = base[q] * (1.0 + 0.01 * n(rng)) + slope[q] * (m - 2);
    T W[5][7];
    for (int m = 0; m < 5; ++m)
      for (int q = 0; q < 7; ++q) W[m][q] = T(w[m][q]);
    hlld += lost(7, 15, [&](const double* g, double* o) {
      T gf[7], a[7], b[7], c = T(0);
      for (int q = 0; q < 7; ++q) gf[q] = T(g[q]), a[q] = b[q] = T(0);
      hlld_vjp<T>(T(5.0 / 3.0), W[1], W[2], T(bn), gf, a, b, c);
      for (int q = 0; q < 7; ++q) o[q] = to_d<T>(a[q]), o[7 + q] = to_d<T>(b[q]);
      o[14] = to_d<T>(c);
    });
    ppmc += lost(14, 36, [&](const double* g, double* o) {
      T gl[7], gr[7], G[5][7], c = T(0);
      for (int q = 0; q < 7; ++q) gl[q] = T(g[q]), gr[q] = T(g[7 + q]);
      for (int q = 0; q < 35; ++q) G[q / 7][q % 7] = T(0);
      ppmc_vjp<T>(T(5.0 / 3.0), T(1e-20), T(1e-20), [&](int m, T* v) { for (int q = 0; q < 7; ++q) v[q] = W[m][q]; }, T(bn),
                  gl, gr, [&](int m, const T* v) { for (int q = 0; q < 7; ++q) G[m][q] = v[q]; }, G[2], c);
      for (int q = 0; q < 35; ++q) o[q] = to_d<T>(G[q / 7][q % 7]);
      o[35] = to_d<T>(c);
    });
    plmc += lost(14, 22, [&](const double* g, double* o) {
      T gl[7], gr[7], G[3][7], c = T(0);
      for (int q = 0; q < 7; ++q) gl[q] = T(g[q]), gr[q] = T(g[7 + q]), G[0][q] = G[1][q] = G[2][q] = T(0);
      plmc_vjp<T>(T(5.0 / 3.0), T(1e-20), T(1e-20), W[1], W[2], W[3], T(bn), gl, gr, G[0], G[1], G[2], c);
      for (int q = 0; q < 21; ++q) o[q] = to_d<T>(G[q / 7][q % 7]);
      o[21] = to_d<T>(c);
    });
  }
  printf("%ld %ld %ld\n", hlld, ppmc, plmc);
}
"""


@pytest.mark.parametrize("typ", ["double", "df"])
def test_nonfinite_cotangents_reach_the_gradient(tmp_path, typ):
    assert compile_and_run(tmp_path, NONFINITE.replace("TYPE", typ)) == ["0", "0", "0"]


CONVERSION = r"""
int main() {
  std::mt19937_64 g(7);
  const uint64_t all = (1ull << 52) - 1;
  long bad = 0;
  for (int i = 0; i < 400000; ++i) {
    uint64_t f = g() & all;
    if (i % 4 == 1) f = ((f >> 29) << 29) + (1ull << 28) + (g() % 3) - 1;  // about halfway between two floats
    if (i % 4 == 2) f = all - (g() & 0xffffffff);                          // hi carries into the exponent
    const int e = i % 4 == 3 ? 944 + (int)(g() % 2) : 944 + (int)(g() % 207);
    if (e == 1150 && f > all - (1ull << 30)) continue;  // rounds to 2^128
    const double x = word_cast<double>(((uint64_t)e << 52) | f) * (g() & 1 ? 1.0 : -1.0);
    const df d = nearest<df>(x);
    bad += !(fabsl(((long double)d.hi - (long double)x) + (long double)d.lo) <= 0x1p-48L * fabsl((long double)x));
    bad += fabs(x - d.hi) != fabs(x - (float)x);       // normalised: hi is x to nearest
  }
  for (double x : values(4)) {
    const df d = nearest<df>(x), t = df_from_double(x);
    const bool tiny = fabs(x) < 0x1p-79, huge = !(fabs(x) < 0x1p127);
    if (tiny) bad += !(fabs((double)d.hi - x) <= fabs(x) * 0x1p-24 + 0x1p-126) + !(fabsf(d.lo) <= 0x1p-100f);
    if (huge) bad += !(d.hi == t.hi || (d.hi != d.hi && t.hi != t.hi) || std::isinf(d.hi));
  }
  printf("%ld\n", bad);
}
"""


def test_float_pairs_of_the_primitives(tmp_path):
    """Within 2^-48 of the double (from_d<df> keeps 2^-47)."""
    assert compile_and_run(tmp_path, CONVERSION) == ["0"]


FALLBACK = r"""
static long used = 0;
int main() {
  std::mt19937_64 g(23);
  std::normal_distribution<double> n;
  std::uniform_real_distribution<double> u;
  long plm = 0, ppm = 0, hl = 0;
  for (int it = 0; it < 40000; ++it) {
    double w[5][7], scale[7], bn = n(g);
    // components and differences of every size, zeros among them
    auto tiny = [&] { return it % 4 == 0 ? 1.0 : u(g) < 0.2 ? 0.0 : std::pow(10.0, -330.0 * u(g)); };
    const double base[7] = {exp(n(g)), n(g), n(g), n(g), exp(n(g)), n(g), n(g)};
    for (double& s : scale) s = tiny();
    bn *= tiny();
    const double size[7] = {1.0, scale[1], scale[2], scale[3], 1.0, scale[5], scale[6]};
    for (int m = 0; m < 5; ++m)
      for (int q = 0; q < 7; ++q) w[m][q] = size[q] * base[q] * (1.0 + 0.05 * scale[(q + 3) % 7] * n(g));
    double a[4][7], b[4][7];
    {
      TryOps<double> o;
      plmc<double>(o, 5.0 / 3.0, w[1], w[2], w[3], bn, a[0], a[1]);
      Ops<double> c;
      plmc<double>(c, 5.0 / 3.0, w[1], w[2], w[3], bn, b[0], b[1]);
      used += o.bad;
      for (int k = 0; k < 14; ++k) plm += !o.bad && !same(a[k / 7][k % 7], b[k / 7][k % 7]);
    }
    {
      TryOps<double> o;
      ppmc<double>(o, 5.0 / 3.0, w, bn, a[0], a[1]);
      Ops<double> c;
      ppmc<double>(c, 5.0 / 3.0, w, bn, b[0], b[1]);
      used += o.bad;
      for (int k = 0; k < 14; ++k) ppm += !o.bad && !same(a[k / 7][k % 7], b[k / 7][k % 7]);
    }
    hlld<double>(5.0 / 3.0, 1.5, w[1], w[2], bn, a[2]);
    Ops<double> c;
    hlld_diff<double>(c, 5.0 / 3.0, 1.5, w[1], w[2], bn, b[2]);
    for (int k = 0; k < 7; ++k) hl += !same(a[2][k], b[2][k]);
  }
  printf("%ld %ld %ld %d\n", plm, ppm, hl, used > 1000);
}
"""


def test_cells_out_of_range_are_flagged(tmp_path):
    """What the range tests let pass equals the complete functions, bit for bit."""
    assert compile_and_run(tmp_path, FALLBACK, flags=("-ffp-contract=off",)) == ["0", "0", "0", "1"]
