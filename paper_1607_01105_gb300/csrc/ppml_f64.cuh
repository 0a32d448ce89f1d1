// FP64 arithmetic of the scheme with as few FP64 instructions as the values allow.
//
// GB300 issues one FP64 warp instruction per 19 cycles and SM (measured: 76 cycles per
// sub-partition against 1 to 2 for a float or integer one), and the FP64 kernels are bound
// by that pipe alone.  The functions below return the very bits of the expressions they
// stand for (round to nearest, no contraction), but take everything that is not an addition,
// a multiplication or a root off the pipe: sign tests, minima, magnitudes and scalings by
// powers of two are integer operations on the words of the number; divisions by a number
// known in advance are one or two multiply-adds with its reciprocal in two parts.  Where an
// operand is out of the range in which that is exact (subnormal, overflowing, NaN), the
// plain expression is evaluated instead, behind a branch that is otherwise not taken.
// 256^3 blast, one step: 96.8 -> 52.1 ms with the integer forms, 14.6 with the shortcuts for
// equal and zero operands; smooth data takes 1294 FP64 instructions a cell instead of 3113.
#pragma once
namespace ppml {
namespace f64 {

__device__ __forceinline__ int hi_word(double x) { return __double2hiint(x); }
__device__ __forceinline__ int lo_word(double x) { return __double2loint(x); }
__device__ __forceinline__ unsigned exponent(double x) {
  return ((unsigned)hi_word(x) >> 20) & 0x7ffu;
}
__device__ __forceinline__ unsigned long long magnitude(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ bool is_zero(double x) {
  return (((unsigned)hi_word(x) << 1) | (unsigned)lo_word(x)) == 0u;
}
__device__ __forceinline__ bool same_bits(double x, double y) {
  return __double_as_longlong(x) == __double_as_longlong(y);
}
__device__ __forceinline__ bool finite(double x) { return exponent(x) != 0x7ffu; }
__device__ __forceinline__ bool positive(double x) {  // x > 0
  const long long b = __double_as_longlong(x);
  return b > 0 && b <= 0x7ff0000000000000ll;
}
// x < b for a positive b
__device__ __forceinline__ bool below(double x, double b) {
  return __double_as_longlong(x) < __double_as_longlong(b) && magnitude(x) <= 0x7ff0000000000000ull;
}
// a normal number with room around it: products and quotients of a few such are normal
__device__ __forceinline__ bool moderate(double x) { return exponent(x) - 623u <= 800u; }

// Plain operations that the compiler does not hoist out of the branch they stand in (a
// speculated FP64 instruction costs what the branch was to save).
#ifdef __CUDA_ARCH__
#define PPML_F64_PLAIN(name, op, expr)                                       \
  __device__ __forceinline__ double name(double a, double b) {               \
    double r;                                                                \
    asm(op " %0, %1, %2;" : "=d"(r) : "d"(a), "d"(b));                       \
    return r;                                                                \
  }
#else
#define PPML_F64_PLAIN(name, op, expr) \
  __device__ __forceinline__ double name(double a, double b) { return expr; }
#endif
PPML_F64_PLAIN(plain_add, "add.rn.f64", a + b)
PPML_F64_PLAIN(plain_sub, "sub.rn.f64", a - b)
PPML_F64_PLAIN(plain_mul, "mul.rn.f64", a * b)
PPML_F64_PLAIN(plain_div, "div.rn.f64", a / b)
#undef PPML_F64_PLAIN

// Uniform and resting gas is common (ambient gas ahead of a blast, the transverse lines of
// planar problems, planes of symmetry), and there most operands are equal or zero.  These
// forms return the value of the plain operation without issuing it then (the sign of a zero
// result may differ, which no later value depends on).
__device__ __forceinline__ double diff(double a, double b) {  // a - b
  if (same_bits(a, b) && finite(a)) return 0.0;
  return plain_sub(a, b);
}
__device__ __forceinline__ double minus(double a, double b) {  // a - b, b often zero
  if (is_zero(b)) return a;
  return plain_sub(a, b);
}
__device__ __forceinline__ double plus(double a, double b) {  // a + b, b often zero
  if (is_zero(b)) return a;
  return plain_add(a, b);
}
__device__ __forceinline__ double times(double a, double b) {  // a b, b often zero
  if (is_zero(b) && finite(a)) return 0.0;
  return plain_mul(a, b);
}
__device__ __forceinline__ double over(double a, double b) {  // a / b, a often zero
  if (is_zero(a) && moderate(b)) return a;
  return plain_div(a, b);
}

// x 2^K by its exponent field where x and the result are normal.
template <int K>
__device__ __forceinline__ double scale(double x) {
  constexpr unsigned lo = K < 0 ? 1 - K : 1, hi = K > 0 ? 2046 - K : 2046;
  if (exponent(x) - lo <= hi - lo)
    return __hiloint2double(hi_word(x) + K * (1 << 20), lo_word(x));
  if (is_zero(x)) return x;
  return plain_mul(x, K < 0 ? 1.0 / (1 << (K < 0 ? -K : 0)) : (double)(1 << (K < 0 ? 0 : K)));
}
__device__ __forceinline__ double half(double x) { return scale<-1>(x); }
__device__ __forceinline__ double twice(double x) { return scale<1>(x); }

// a b > 0, as the rounded product says it.
__device__ __forceinline__ bool product_positive(double a, double b) {
  const unsigned ea = exponent(a), eb = exponent(b);
  if ((hi_word(a) ^ hi_word(b)) < 0) return false;  // negative, a zero or NaN
  if (ea - 1u < 2046u && eb - 1u < 2046u && ea + eb >= 972u) return true;  // normal, no underflow
  if (is_zero(a) || is_zero(b)) return false;
  return plain_mul(a, b) > 0.0;
}
// a b <= 0 (false if the product is NaN).
__device__ __forceinline__ bool product_nonpositive(double a, double b) {
  const unsigned ea = exponent(a), eb = exponent(b);
  if (ea < 2047u && eb < 2047u) {
    if ((hi_word(a) ^ hi_word(b)) < 0) return true;
    if (ea != 0u && eb != 0u && ea + eb >= 972u) return false;
    if (is_zero(a) || is_zero(b)) return true;
  }
  return plain_mul(a, b) <= 0.0;
}

// x / 3 and x / 6: x zl + x zh with the reciprocal in two parts (Brisebarre, Muller and
// Raina, "Accelerating correctly rounded floating-point division when the divisor is known
// in advance", 2004).  A quotient by 3 lies at least 1/6 of its last place from every
// midpoint of two doubles (2 X 2^s and 3 (2 k + 1) differ in parity), and the sum before
// its rounding is within 2^-100 of the quotient, so the rounding is the quotient's.  Below
// 2^-959 the low product underflows.
__device__ __forceinline__ double div3(double x) {
  if (exponent(x) < 64u && !is_zero(x)) return plain_div(x, 3.0);
  constexpr double zh = 0x1.5555555555555p-2, zl = 0x1.5555555555555p-56;  // 1/3
  return __fma_rn(x, zh, __dmul_rn(x, zl));
}
__device__ __forceinline__ double div6(double x) {
  if (exponent(x) < 64u && !is_zero(x)) return plain_div(x, 6.0);
  constexpr double zh = 0x1.5555555555555p-3, zl = 0x1.5555555555555p-57;  // 1/6
  return __fma_rn(x, zh, __dmul_rn(x, zl));
}

// A divisor known in advance: h with its reciprocal in two parts (zh = 1/h rounded, zh + zl
// = 1/h to 2^-104).  safe: h's exponent leaves room for the intermediate products.
struct Divisor {
  double h, zh, zl;
};
__device__ __forceinline__ Divisor divisor(double h) {
  Divisor d;
  d.h = h;
  d.zh = 1.0 / h;
  d.zl = __dmul_rn(__fma_rn(-d.zh, h, 1.0), d.zh);
  return d;
}
// x / d.h: x zh + x zl is within a last place of the quotient, its remainder is exact, and
// one correction with the rounded reciprocal rounds correctly (Markstein, "Computation of
// elementary functions on the IBM RISC System/6000 processor", 1990).
__device__ __forceinline__ double divide(double x, const Divisor& d) {
  const unsigned ex = exponent(x), eh = exponent(d.h);
  if (ex - 400u <= 1200u && eh - 823u <= 400u) {
    const double q = __fma_rn(x, d.zh, __dmul_rn(x, d.zl));
    return __fma_rn(__fma_rn(-q, d.h, x), d.zh, q);
  }
  if (is_zero(x) && eh - 1u < 2046u) return x;  // (the divisors are positive)
  return plain_div(x, d.h);
}

// Appendix, Step 1 from the differences l = q0 - qm, r = qp - q0: the limited slope
// min(|w| / 2, 2 |l|, 2 |r|) with the sign of w = qp - qm, 0 unless l r > 0 (then none of
// them is NaN and magnitudes order as integers).
__device__ __forceinline__ double slope(double l, double r, double qm, double qp) {
  if (!product_positive(r, l)) return 0.0;
  const double w = plain_sub(qp, qm);
  const unsigned long long ml = magnitude(l), mr = magnitude(r);
  const double m2 = twice(__longlong_as_double((long long)(ml < mr ? ml : mr)));
  const double dq = half(w);
  const unsigned long long a = magnitude(dq), b = magnitude(m2), m = a < b ? a : b;
  return __longlong_as_double(
      (long long)(m | ((unsigned long long)__double_as_longlong(dq) & 0x8000000000000000ull)));
}

// Appendix, Step 1: the face value (q0 + q1) / 2 - (d1 - d0) / 6.
__device__ __forceinline__ double face(double q0, double q1, double d0, double d1) {
  if (is_zero(d0) && is_zero(d1)) {
    if (same_bits(q0, q1) && exponent(q0) < 2046u) return q0;
    return half(plain_add(q0, q1));
  }
  return plain_sub(half(plain_add(q0, q1)), div6(plain_sub(d1, d0)));
}

// Appendix, Steps 2-3: whether the unflattened parabola (D, S) overshoots: 1 if D S > D D
// (the left face is moved), -1 if D S < -D D (the right one), else 0.  |S| <= |D| is
// neither, as rounding is monotone; |S| at least four last places above |D| with products
// in the normal range is one of the two, by the signs.
__device__ __forceinline__ int overshoot(double D, double S) {
  const unsigned long long a = magnitude(D), b = magnitude(S);
  if (b <= a && b < 0x7ff0000000000000ull && a < 0x7ff0000000000000ull) return 0;
  if (b >= a + 4u && a >= (550ull << 52) && b < (1450ull << 52))
    return (hi_word(D) ^ hi_word(S)) < 0 ? -1 : 1;
  const double ds = plain_mul(D, S), dd = plain_mul(D, D);
  return ds > dd ? 1 : (ds < -dd ? -1 : 0);
}

// Appendix, Steps 2-3: a cell's parabola (faces L, R, D = R - L and S = q^(6)) from its value
// and its two unlimited faces, in place.
__device__ __forceinline__ void parabola(double q0, double& L, double& R, double& D, double& S) {
  if (product_nonpositive(diff(L, q0), diff(q0, R))) {  // flat
    L = R = q0;
    D = S = 0.0;  // q0 - q0 and 6 (q0 - q0)
    if (!finite(q0)) D = S = plain_sub(q0, q0);
    return;
  }
  D = plain_sub(R, L);
  S = plain_mul(6.0, plain_sub(q0, half(plain_add(L, R))));
  const int o = overshoot(D, S);
  if (o != 0) {
    if (o > 0)
      L = plain_sub(plain_mul(3.0, q0), twice(R));
    else
      R = plain_sub(plain_mul(3.0, q0), twice(L));
    D = plain_sub(R, L);
    S = plain_mul(6.0, plain_sub(q0, half(plain_add(L, R))));
  }
}

// What the characteristic averages read of a Courant number y: y / 2 and 1 - 2 y / 3.
struct Weights {
  double hy, w;
};
__device__ __forceinline__ Weights weights(double y) {
  Weights k;
  k.hy = half(y);
  k.w = is_zero(y) ? 1.0 : plain_sub(1.0, div3(twice(y)));
  return k;
}
// Average next to the right face of a cell (face value F = R, sgn -1: R - y/2 (D - S w)) or
// to its left one (F = L, sgn +1: L + y/2 (D + S w)); adding a negated term is subtracting.
__device__ __forceinline__ double average(bool right, double F, double D, double S,
                                          const Weights& k) {
  if (is_zero(D) && is_zero(S)) return F;
  const double t = plain_mul(S, k.w);
  const double u = plain_mul(k.hy, plain_add(D, right ? -t : t));
  return plain_add(F, right ? -u : u);
}

}  // namespace f64
}  // namespace ppml
