"""The FP64 helper functions of the kernels (ppml_f64.cuh), compiled for the host, return the
bits of the plain expressions they stand for: random operands over many exponents, and
zeros, subnormals, overflowing values, infinities and NaN."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1607_01105_gb300", "csrc")

HARNESS = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <limits>
#define __device__
#define __forceinline__ inline
static inline double bits(uint64_t u) { double d; memcpy(&d, &u, 8); return d; }
static inline uint64_t word(double d) { uint64_t u; memcpy(&u, &d, 8); return u; }
static inline int __double2hiint(double x) { return (int)(word(x) >> 32); }
static inline int __double2loint(double x) { return (int)word(x); }
static inline double __hiloint2double(int h, int l) { return bits(((uint64_t)(uint32_t)h << 32) | (uint32_t)l); }
static inline long long __double_as_longlong(double x) { return (long long)word(x); }
static inline double __longlong_as_double(long long x) { return bits((uint64_t)x); }
static inline double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
static inline double __dmul_rn(double a, double b) { return a * b; }
#include "ppml_f64.cuh"
using namespace ppml::f64;
static uint64_t s = 88172645463325252ull;
static uint64_t rnd() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s * 2685821657736338717ull; }
static double draw(int kind) {
  static const double special[] = {0.0, -0.0, 1.0, -1.0, 3.0, 6.0, 5e-324, -5e-324, 1e-310, 2.2250738585072014e-308,
      1.7976931348623157e308, -1.7976931348623157e308, std::numeric_limits<double>::infinity(),
      -std::numeric_limits<double>::infinity(), std::numeric_limits<double>::quiet_NaN(), 1e-200, 1e200, 1e-160, -1e-160};
  uint64_t r = rnd();
  if (kind == 0) return special[r % (sizeof(special) / sizeof(special[0]))];
  if (kind == 1) return bits(r);                                                  // any exponent
  return bits((r & 0x800fffffffffffffull) | ((1023 - 8 + rnd() % 17) << 52));      // near 1
}
static bool same(double a, double b) { return (a != a && b != b) || word(a) == word(b); }
static int bad = 0;
#define CHECK(name, got, want) do { double g = (got), w = (want); if (!same(g, w)) { if (bad++ < 20) printf("%s: %a %a gave %a, is %a\n", name, x, y, g, w); } } while (0)
int main() {
  for (long n = 0; n < 6000000; n++) {
    const int ka = n % 16 == 0 ? 0 : (n % 4 == 1 ? 1 : 2), kb = n % 11 == 0 ? 0 : (n % 5 == 1 ? 1 : 2);
    double x = draw(ka), y = draw(kb), z = draw(kb);
    if (n % 3 == 0) y = bits(word(x) + (rnd() % 17) - 8);  // neighbours of x
    if (n % 7 == 0) z = -y;
    CHECK("half", half(x), 0.5 * x);
    CHECK("twice", twice(x), 2.0 * x);
    CHECK("scale -4", scale<-4>(x), x / 16.0);
    CHECK("scale -3", scale<-3>(x), x / 8.0);
    CHECK("div3", div3(x), x / 3.0);
    CHECK("div6", div6(x), x / 6.0);
    CHECK("divide", divide(x, divisor(std::fabs(y))), x / std::fabs(y));
    CHECK("positive", product_positive(x, y), x * y > 0.0);
    CHECK("nonpositive", product_nonpositive(x, y), x * y <= 0.0);
    const double l = y - x, r = z - y, dq = 0.5 * (z - x);
    const double m = std::fmin(std::fabs(dq), 2.0 * std::fmin(std::fabs(r), std::fabs(l)));
    CHECK("slope", slope(l, r, x, z), r * l > 0.0 ? std::copysign(m, dq) : 0.0);
    // equal up to the sign of a zero
    CHECK("diff", diff(x, y) + 0.0, (x - y) + 0.0);
    CHECK("plus", plus(x, n % 9 ? y : 0.0) + 0.0, (x + (n % 9 ? y : 0.0)) + 0.0);
    CHECK("minus", minus(x, n % 9 ? y : 0.0) + 0.0, (x - (n % 9 ? y : 0.0)) + 0.0);
    CHECK("times", times(x, n % 9 ? y : 0.0) + 0.0, (x * (n % 9 ? y : 0.0)) + 0.0);
    CHECK("over", over(n % 9 ? x : 0.0, y) + 0.0, ((n % 9 ? x : 0.0) / y) + 0.0);
    CHECK("positive value", positive(x), x > 0.0);
    CHECK("below", below(x, 1.5), x < 1.5);
    const double d0 = n % 2 ? 0.0 : r, d1 = n % 2 ? 0.0 : l, yy = n % 6 == 3 ? x : y;
    CHECK("face", face(x, yy, d0, d1) + 0.0, (0.5 * (x + yy) - (d1 - d0) / 6.0) + 0.0);
    {
      double L = 0.5 * (x + y) - l / 6.0, R = 0.5 * (y + z) - r / 6.0, D, S;  // cell value y
      const double L0 = L, R0 = R;
      parabola(y, L, R, D, S);
      double Ln = L0, Rn = R0;
      if ((L0 - y) * (y - R0) <= 0.0) {
        Ln = Rn = y;
      } else {
        const double d = R0 - L0, q6 = 6.0 * (y - 0.5 * (L0 + R0));
        if (d * q6 > d * d) Ln = 3.0 * y - 2.0 * R0;
        else if (d * q6 < -(d * d)) Rn = 3.0 * y - 2.0 * L0;
      }
      const double Dn = Rn - Ln, Sn = 6.0 * (y - 0.5 * (Ln + Rn));
      const bool huge = std::fabs(y) > 8e307;  // y + y overflows
      if (!huge) {
        CHECK("parabola L", L, Ln);
        CHECK("parabola R", R, Rn);
        CHECK("parabola D", D + 0.0, Dn + 0.0);
        CHECK("parabola S", S + 0.0, Sn + 0.0);
        const double c = 0.3;
        const Weights k = weights(c);
        CHECK("right average", average(true, R, D, S, k) + 0.0, (Rn - 0.5 * c * (Dn - Sn * (1.0 - 2.0 * c / 3.0))) + 0.0);
        CHECK("left average", average(false, L, D, S, k) + 0.0, (Ln + 0.5 * c * (Dn + Sn * (1.0 - 2.0 * c / 3.0))) + 0.0);
      }
    }
    CHECK("overshoot", overshoot(x, y), x * y > x * x ? 1 : (x * y < -(x * x) ? -1 : 0));
  }
  printf("%d wrong\n", bad);
  return bad != 0;
}
"""


@pytest.mark.parametrize("flags", [["-O2"], ["-O0"]])
def test_f64_helpers_return_the_bits_of_the_plain_expressions(tmp_path, flags):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(HARNESS)
    subprocess.check_call([gxx, "-std=c++17", "-ffp-contract=off", *flags, f"-I{CSRC}", str(src), "-o", str(exe)])
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stdout
