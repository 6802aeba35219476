"""The double-float arithmetic of the FP32 inner solves (fct_df.cuh), compiled for
the host: exact squares and two-sums, products, sums of positive terms and quotients
within 2^-44, and comparisons that see what a pair's low word says (a residual that
falls by less than one part in 2^24 has still fallen; a squared tolerance is met to
the pair's precision)."""
import shutil
import subprocess

import pytest

from paper_2309_14584_gb300 import build as B

SOURCE = r"""
#include "fct_df.cuh"
#include <cstdio>
#include <random>

static long double val(float2 a) { return static_cast<long double>(a.x) + a.y; }
static int bad = 0;
static void check(bool ok, const char* what, double a, double b) {
  if (!ok && ++bad < 10) std::printf("%s: %.17g %.17g\n", what, a, b);
}

int main() {
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> mant(1.0, 2.0), expo(-30.0, 30.0);
  auto draw = [&] { return std::ldexp(mant(g), static_cast<int>(expo(g))); };
  const long double eps = std::ldexp(1.0L, -44);
  for (int i = 0; i < 200000; ++i) {
    const double a = draw(), b = draw();
    const float2 fa = df_of(a), fb = df_of(b);
    check(std::fabs(val(fa) - a) <= std::ldexp(1.0L, -47) * a, "of", a, 0);
    const float t = static_cast<float>(a);
    check(val(df_square(t)) == static_cast<long double>(t) * t, "square", t, 0);
    const float2 ts = df_two_sum(t, static_cast<float>(-b));
    check(val(ts) == static_cast<long double>(t) - static_cast<float>(b), "two_sum", a, b);
    const long double s = val(fa) + val(fb), p = val(fa) * val(fb), q = val(fa) / val(fb);
    check(std::fabs(val(df_add(fa, fb)) - s) <= eps * s, "add", a, b);
    check(std::fabs(val(df_mul(fa, fb)) - p) <= eps * p, "mul", a, b);
    check(std::fabs(val(df_div(fa, fb)) - q) <= eps * q, "div", a, b);
    // the rounded quotient is within half a unit of FP32 of the exact one, but for 2^-19 of a unit
    const float al = df_div(fa, fb).x;
    const float up = std::nextafterf(al, 3e38f);
    check(std::fabs(al - q) <= (0.5L + std::ldexp(1.0L, -19)) * (static_cast<long double>(up) - al), "alpha", a, b);
    // comparisons: as those of the values
    const double near = a * (1.0 + std::ldexp(mant(g) - 1.5, -25));
    const float2 fn = df_of(near);
    check(df_less(fa, fn) == (val(fa) < val(fn)), "less", a, near);
    check(df_less(fn, fa) == (val(fn) < val(fa)), "less", near, a);
    check(!df_less(fa, fa), "less itself", a, a);
    check(df_less(fa, fb) == (val(fa) < val(fb)), "less far", a, b);
  }
  const float2 one = df_of(1.0), below = df_of(1.0 - std::ldexp(1.0, -40));
  check(df_less(below, one) && !df_less(one, below), "one", 1.0, 0.0);
  std::printf("%d\n", bad);
  return bad != 0;
}
"""


def test_rounding_and_comparisons(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    src = tmp_path / "df.cpp"
    src.write_text(SOURCE)
    exe = tmp_path / "df"
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-x", "c++", "-I", B.CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], stdout=subprocess.PIPE, text=True)
    assert r.returncode == 0, r.stdout
