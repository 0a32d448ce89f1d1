// Device building blocks of the PPML step (Kulikov & Vorobyov, arXiv:1607.01105),
// templated on the arithmetic type T (float or double).  Each helper states the passage
// it implements.  Readings of garbled or silent passages (identical to the ones the
// project's independent CPU oracle takes):
//   * Delta q = q^R - q^L (Appendix prints q^L - q^R, contradicting eq. A1 and the
//     characteristic averages);
//   * rho_L, rho_R, p_L, p_R inside the Roe averages, lambda and the impedance are the
//     adjacent cell values; only v and p carrying (-+ lambda t) are parabola averages;
//   * the monotonicity step tests "flat" first, then applies at most one overshoot fix.
//
// Precision policy.  The double instantiation is compiled without FMA contraction and
// evaluates every expression in the same order as the FP64 oracle (x/6, 2y/3,
// (speed * tau) / h), so the FP64 path reproduces it bit for bit.  The float
// instantiation uses the cheaper forms (doubled slopes, x * (1/12), y * (2/3),
// speed * (tau/h)) and FMAs.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "ppml_f64.cuh"

namespace ppml {

// Constants of a sweep along one axis: tau, h, th = tau / h (and FP64: 1 / h).
template <typename T>
struct AxisStep;

template <>
struct AxisStep<float> {
  float th;
  __device__ __forceinline__ AxisStep(double, const f64::Divisor&, float th_) : th(th_) {}
};
template <>
struct AxisStep<double> {
  double th, tau;
  f64::Divisor h;
  __device__ __forceinline__ AxisStep(double tau_, const f64::Divisor& h_, double th_)
      : th(th_), tau(tau_), h(h_) {}
};

// Courant number s tau / h of a signal speed s (FP32: with th = tau / h precomputed).
__device__ __forceinline__ float courant(float s, const AxisStep<float>& k) { return s * k.th; }
__device__ __forceinline__ double courant(double s, const AxisStep<double>& k) {
  return f64::divide(s * k.tau, k.h);
}

template <typename T>
struct Parab {
  T L, R, D, S;  // q^L, q^R, Delta q = q^R - q^L, q^(6)
};

__device__ __forceinline__ float tabs(float x) { return x < 0.0f ? -x : x; }
__device__ __forceinline__ double tabs(double x) { return fabs(x); }
// Sums and differences whose second operand is often zero in FP64 (f64::plus, minus).
__device__ __forceinline__ float sub_term(float a, float b) { return a - b; }
__device__ __forceinline__ double sub_term(double a, double b) { return f64::minus(a, b); }
__device__ __forceinline__ float add_term(float a, float b) { return a + b; }
__device__ __forceinline__ double add_term(double a, double b) { return f64::plus(a, b); }

// Appendix, Step 1: limited slope delta_m q_i.  Branch-free: min(|dq|, 2 min(|r|, |l|))
// equals min(|dq|, 2|r|, 2|l|) exactly (doubling is exact), and r l > 0 implies q is
// strictly monotone, so dq != 0 (up to underflow to a zero of either sign) and the sign
// copy equals the test dq > 0; where r l <= 0 the result is +0 whatever the signs of the
// zeros inside, so fabs (an operand modifier) gives the values of the sign test.
// The FP32 instantiation returns twice the slope, min(|q+ - q-|, 4|r|, 4|l|) with its sign
// (every scaling exact), which face_value expects: the halving is folded into its 1/6.
template <typename T>
__device__ __forceinline__ T limited_slope(T qm, T q0, T qp) {
  if constexpr (sizeof(T) == 8) {
    const T r = f64::diff(qp, q0), l = f64::diff(q0, qm);
    return f64::slope(l, r, qm, qp);
  } else {
    const T r = qp - q0, l = q0 - qm;
    const T dq2 = qp - qm;
    const T m2 = fmin(fabs(dq2), T(4) * fmin(fabs(r), fabs(l)));
    return r * l > T(0) ? copysign(m2, dq2) : T(0);
  }
}

// Appendix, Step 1: 4th-order face value q_{i+1/2} from the cell values and limited slopes
// (FP32: from the doubled slopes of limited_slope, (d1 - d0) / 12 = the (d1 - d0) / 6 of
// the halved values).
template <typename T>
__device__ __forceinline__ T face_value(T q0, T q1, T d0, T d1) {
  if constexpr (sizeof(T) == 8)
    return f64::face(q0, q1, d0, d1);
  else
    return T(0.5) * (q0 + q1) - (d1 - d0) * (1.0f / 12.0f);
}

// Appendix, Steps 2-3: parabola of a cell from its value and its two face values.
// Branch-free: the overshoot tests are evaluated on the unflattened faces and only
// selected when the cell is not flattened, which gives the same values as the
// sequential form (flat test first, then at most one fix).
template <typename T>
__device__ __forceinline__ Parab<T> parabola(T q0, T L, T R) {
  if constexpr (sizeof(T) == 8) {
    Parab<T> p;
    p.L = L;
    p.R = R;
    f64::parabola(q0, p.L, p.R, p.D, p.S);
    return p;
  }
  const bool flat = (L - q0) * (q0 - R) <= T(0);
  const T D = R - L;
  const T S = T(6) * (q0 - T(0.5) * (L + R));
  // at most one fix: D S > D D >= 0 >= -(D D) excludes D S < -(D D)
  const bool fixL = D * S > D * D;
  const bool fixR = D * S < -(D * D);
  const T Ln = flat ? q0 : (fixL ? T(3) * q0 - T(2) * R : L);
  const T Rn = flat ? q0 : (fixR ? T(3) * q0 - T(2) * L : R);
  Parab<T> p;
  p.L = Ln;
  p.R = Rn;
  p.D = Rn - Ln;
  p.S = T(6) * (q0 - T(0.5) * (Ln + Rn));
  return p;
}

// Appendix, characteristic integrals: mean of the parabola over the right fraction y of
// the cell (q_L(-lambda t), y = lambda t / h; FP64: f64::average) ...
__device__ __forceinline__ float avg_right(float R, float D, float S, float y) {
  return R - 0.5f * y * (D - S * (1.0f - y * (2.0f / 3.0f)));
}
// ... and over its left fraction y (q_R(lambda t)).
__device__ __forceinline__ float avg_left(float L, float D, float S, float y) {
  return L + 0.5f * y * (D + S * (1.0f - y * (2.0f / 3.0f)));
}

// Sec. 1.1/1.2: face constants of the acoustic Riemann problem from the adjacent cell
// values: lambda = sqrt(gamma p^/rho^) and the impedance Z = rho^ lambda (FP64; sl, sr the
// square roots of rl, rr, and ws the products rho sqrt(rho), p sqrt(rho) of a cell, each
// formed once per cell by the caller).
struct RootWeights {
  double s, a, b;  // sqrt(rho), rho sqrt(rho), p sqrt(rho)
};
__device__ __forceinline__ RootWeights root_weights(double rho, double p) {
  RootWeights w;
  w.s = sqrt(rho);
  w.a = rho * w.s;
  w.b = p * w.s;
  return w;
}
// A cell between whose faces nothing varies: rho and p positive, mid-range.
__device__ __forceinline__ bool plain_gas(double rho, double p) {
  return f64::hi_word(rho) >= 0 && f64::hi_word(p) >= 0 && f64::moderate(rho) && f64::moderate(p);
}
__device__ __forceinline__ void face_constants(const RootWeights& l, const RootWeights& r,
                                               double gamma, double& lam, double& Z) {
  const double A = l.a + r.a;  // rho_L^{3/2} + rho_R^{3/2}
  const double B = l.b + r.b;  // p_L sqrt(rho_L) + p_R sqrt(rho_R)
  const double S = l.s + r.s;
  lam = sqrt(gamma * B / A);
  Z = sqrt(gamma * A * B / (S * S));
}

// eqs. lowriemannvelocity / lowriemannpressure from the four characteristic averages.
__device__ __forceinline__ void riemann_vp(double vls, double vrs, double pls, double prs,
                                           double Z, double& V, double& P) {
  V = f64::half(vls + vrs) + (pls - prs) / f64::twice(Z);
  P = f64::half(pls + prs) + f64::half(Z) * (vls - vrs);
}

// Sec. 1.4: energy consistency of one cell, in double.  u = {rho, mx, my, mz, rhoE, rhoeps}.
// Returns 1 if the cell took the vacuum branch.  PLAIN: without the shortcuts for zero
// operands.
template <bool PLAIN>
__device__ __forceinline__ int energy_correction(double u[6], double rho_vac) {
  const double rho = u[0];
  double m2;
  if constexpr (PLAIN) {
    m2 = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
  } else {
    if (f64::is_zero(u[1]) && f64::is_zero(u[2]) && f64::is_zero(u[3]) && f64::moderate(rho)) {
      if (f64::positive(u[4])) u[5] = u[4];  // at rest: rho E - 0 / (2 rho)
      return 0;
    }
    m2 = f64::plus(f64::plus(u[1] * u[1], f64::times(u[2], u[2])), f64::times(u[3], u[3]));
  }
  if (f64::below(rho, rho_vac) && f64::positive(m2)) {
    const double de = u[4] - u[5];
    if (de < 0.0) {
      u[1] = u[2] = u[3] = 0.0;
      u[5] = u[4];
      return 1;
    }
    const double vnew = sqrt(2.0 * de / rho);
    const double vold = sqrt(m2) / rho;
    const double s = vnew / vold;
    u[1] *= s;
    u[2] *= s;
    u[3] *= s;
    return 1;
  }
  const double e = u[4] - m2 / (PLAIN ? 2.0 * rho : f64::twice(rho));
  if (f64::positive(e)) u[5] = e;
  return 0;
}

// ------------------------------------------------------- approximate FP32 operations
// PTX rcp.approx.f32 / sqrt.approx.f32 (relative error about 2^-23, one special-function
// instruction each).  The FP32 stage kernels use them where the result only feeds
// tolerance-checked FP32 arithmetic (velocities m / rho, Roe weights, the acoustic face
// constants, signal speeds); the FP64 instantiation never does.
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// FP32 face constants (as face_constants) from the adjacent cell values and their square
// roots sl, sr (computed once per cell by the caller): lambda = sqrt(gamma B / A) and
// Z = sqrt(gamma A B) / S = lambda A / S.  Also returns 1 / (2 Z) for the velocity.
__device__ __forceinline__ void face_constants_f32(float rl, float rr, float sl, float sr,
                                                   float pl, float pr, float gamma, float& lam,
                                                   float& Z, float& half_rz) {
  const float A = rl * sl + rr * sr;
  const float B = pl * sl + pr * sr;
  const float S = sl + sr;
  lam = sqrt_approx(gamma * B * rcp_approx(A));
  Z = lam * A * rcp_approx(S);
  half_rz = 0.5f * rcp_approx(Z);
}

// ------------------------------------------------- FP32 parabolas in deviation form
// The plain FP32 kernels (line pipelines in ppml_pair.cuh) carry a cell's parabola as its two
// face deviations from the cell value,
// l = q0 - q^L and r = q^R - q0 (stored doubled), instead of (q^L, q^R, Delta q, q^(6)):
//   * the monotonicity step (Appendix, Steps 2-3) reads, with Delta q = l + r and
//     q^(6) = 3 (l - r): flat where l r <= 0, else l <- min(|l|, 2|r|) and
//     r <- min(|r|, 2|l|) with their signs (the overshoot tests Delta q q^(6) > Delta q^2
//     and < -Delta q^2 are |l| > 2|r| and |r| > 2|l|);
//   * the characteristic averages (Appendix) of the part y = lambda t / h next to a face
//     become q0 + (1-y)^2 r + y (1-y) l on the cell's right side and
//     q0 - (1-y)^2 l - y (1-y) r on its left side.
// The same functions of the cell values with a third of the operations, and the deviations
// are formed from differences of neighbouring cells, so they carry no rounding of q itself.
// The limited slope is |.| and sign arithmetic of the two differences as well: PTX
// min.xorsign.abs returns the smaller magnitude with the product of the signs.
__device__ __forceinline__ float min_xs(float a, float b) {
  float r;
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
// the same, NaN if either operand is (a non-finite face makes the cell's parabola NaN)
__device__ __forceinline__ float min_xs_nan(float a, float b) {
  float r;
  asm("min.NaN.xorsign.abs.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// Weights of the deviations at Courant number y, halved for the doubled deviations.
struct DevWeights {
  float a, b;  // (1-y)^2 / 2, y (1-y) / 2
};
__device__ __forceinline__ DevWeights dev_weights(float y) {
  const float z = 1.0f - y, hz = 0.5f * z;
  DevWeights w;
  w.a = hz * z;
  w.b = hz * y;
  return w;
}
// ---------------------------------------------------------- compensated FP32 helpers
// Error-free transformations (Knuth TwoSum; FMA-based TwoProduct).  Used where the
// paper's quantity is a small difference of large totals so that the FP32 path keeps
// FP64-class accuracy without GB300's reduced-rate FP64 pipe.

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// rho eps = rho E - |m|^2 / (2 rho) evaluated in double-float (about 44 significant
// bits) and rounded once to float.  Sec. 1.4 (dense branch).
__device__ __forceinline__ float internal_energy_ff(float rho, float mx, float my, float mz,
                                                    float en) {
  const float p1 = mx * mx, e1 = fmaf(mx, mx, -p1);
  const float p2 = my * my, e2 = fmaf(my, my, -p2);
  const float p3 = mz * mz, e3 = fmaf(mz, mz, -p3);
  float s, t1, hi, t2;
  two_sum(p1, p2, s, t1);
  two_sum(s, p3, hi, t2);
  const float lo = ((t1 + t2) + (e1 + e2)) + e3;  // |m|^2 = hi + lo
  const float r2 = 2.0f * rho;
  const float ir2 = rcp_approx(r2);
  const float q = hi * ir2;
  const float rem = fmaf(-q, r2, hi) + lo;  // remainder of hi (exact to 2^-46) plus lo
  const float ql = rem * ir2;               // |m|^2/(2 rho) = q + ql
  float d, de;
  two_sum(en, -q, d, de);
  return d + (de - ql);
}

// The same with one momentum component (the operations that are left when the others are 0).
__device__ __forceinline__ float internal_energy_1d(float rho, float m, float en) {
  const float hi = m * m, lo = fmaf(m, m, -hi);
  const float r2 = 2.0f * rho, ir2 = rcp_approx(r2);
  const float q = hi * ir2;
  const float ql = (fmaf(-q, r2, hi) + lo) * ir2;
  float d, de;
  two_sum(en, -q, d, de);
  return d + (de - ql);
}

// ------------------------------------------------------------ double-float state values
// A field stored as an unevaluated float pair (hi, lo), |lo| <= ulp(hi) / 2, carries about
// 48 significant bits.  The FP32 path keeps rho, m and rho E this way when the caller
// supplies the low parts: the stencil arithmetic reads hi, and every update of a stored
// value and the Sec. 1.4 difference rho E - |m|^2 / (2 rho) use both parts.

// (hi, lo) = (h + l) - d, renormalised (TwoSum of h and -d, then the low terms).
__device__ __forceinline__ void df_sub(float h, float l, float d, float& hi, float& lo) {
  float s, e;
  two_sum(h, -d, s, e);
  e += l;
  hi = s + e;
  lo = e - (hi - s);
}

// Split a double into its float pair.
__device__ __forceinline__ void df_split(double x, float& hi, float& lo) {
  hi = (float)x;
  lo = (float)(x - (double)hi);
}

// Quotients by a divisor known at launch, for 0 <= n < 2^31 (any cell index): n m >> s with
// m = 2^s / d rounded up and s = 31 + ceil(log2 d), whose error n (m d - 2^s) < 2^s leaves the
// quotient's integer part (Granlund and Montgomery, "Division by invariant integers using
// multiplication", 1994).  A 64-bit division takes some 60 instructions, this three.
struct IndexDivisor {
  unsigned m;
  int s;
  explicit IndexDivisor(int d) {
    int l = 0;
    while ((1ll << l) < d) l++;
    s = 31 + l;
    m = (unsigned)((1ull << s) / (unsigned)d + 1u);
  }
  __host__ __device__ unsigned quotient(unsigned n) const {
    return (unsigned)(((unsigned long long)n * m) >> s);
  }
};

// A value of a host-formed table as a kernel of either precision reads it: the double
// itself, or its float pair (hi, lo).
struct FloatPair {
  float x, y;
};
template <typename T>
struct TableOf {
  using type = double;
};
template <>
struct TableOf<float> {
  using type = FloatPair;
};
// A table value in the arithmetic V of the kernel that reads it.
template <typename V, typename U>
__device__ __forceinline__ V table_as(U t) {
  if constexpr (std::is_same_v<V, U>)
    return t;
  else
    return (double)t.x + (double)t.y;
}

// c / (1 - p t) of the Poisson symbols: p the product of two tables, t the third.  In float
// pairs every product and the difference keep about 2^-46, so 1 - p t of the smoothest mode
// of N points, about (4/3)(pi / N)^2, keeps 30 bits at N = 512, more than the float
// amplitude it scales; the quotient takes one Newton correction.  (FP64 would take some 15
// instructions at one per 19 cycles and SM.)
__device__ __forceinline__ double table_product(double a, double b) { return a * b; }
__device__ __forceinline__ FloatPair table_product(FloatPair a, FloatPair b) {
  const float p = a.x * b.x;
  const float e = fmaf(a.x, b.x, -p) + fmaf(a.x, b.y, a.y * b.x);
  FloatPair r;
  r.x = p + e;
  r.y = (p - r.x) + e;
  return r;
}
__device__ __forceinline__ double over_one_minus(double c, double p, double t) {
  return c / (1.0 - p * t);
}
__device__ __forceinline__ FloatPair over_one_minus(FloatPair c, FloatPair p, FloatPair t) {
  const float q = p.x * t.x;
  const float qe = fmaf(p.x, t.x, -q) + fmaf(p.x, t.y, p.y * t.x);
  float d, de;
  two_sum(1.0f, -q, d, de);
  const float l = de - qe;
  const float dh = d + l, dl = (d - dh) + l;  // 1 - p t
  const float r = rcp_approx(dh);
  FloatPair f;
  f.x = c.x * r;
  f.y = (fmaf(-f.x, dh, c.x) + fmaf(-f.x, dl, c.y)) * r;
  return f;
}
__device__ __forceinline__ double scaled(double v, double f) { return v * f; }
__device__ __forceinline__ float scaled(float v, FloatPair f) { return fmaf(v, f.x, v * f.y); }
__device__ __forceinline__ float scaled(float v, double f) { return (float)((double)v * f); }

// rho eps = (eh + el) - |m|^2 / (2 rho) with rho = rh + rl and m_a = mh_a + ml_a, in
// double-float (about 44 significant bits), rounded once to float.  Sec. 1.4 (dense
// branch) on double-float totals: the error of the difference does not grow with the
// ratio of kinetic to internal energy beyond the double-float rounding.
__device__ __forceinline__ float internal_energy_df(float rh, float rl, const float mh[3],
                                                    const float ml[3], float eh, float el) {
  float p[3], e[3];
#pragma unroll
  for (int a = 0; a < 3; a++) {
    p[a] = mh[a] * mh[a];
    e[a] = fmaf(mh[a], mh[a], -p[a]) + 2.0f * mh[a] * ml[a];  // ml^2 is below 2^-48 |m|^2
  }
  float s, t1, hi, t2;
  two_sum(p[0], p[1], s, t1);
  two_sum(s, p[2], hi, t2);
  const float lo = ((t1 + t2) + (e[0] + e[1])) + e[2];  // |m|^2 = hi + lo
  const float r2 = 2.0f * rh, r2l = 2.0f * rl;            // 2 rho = r2 + r2l exactly
  const float ir2 = rcp_approx(r2);
  const float q = hi * ir2;
  const float rem = (fmaf(-q, r2, hi) - q * r2l) + lo;  // hi + lo - q (r2 + r2l)
  const float ql = rem * ir2;                           // |m|^2 / (2 rho) = q + ql
  float d, de;
  two_sum(eh, -q, d, de);
  return d + ((de + el) - ql);
}

// Neumaier-compensated running sum in float; value() = hi + lo in double.
struct CompSum {
  float hi, lo;
  __device__ __forceinline__ void init() { hi = 0.f; lo = 0.f; }
  __device__ __forceinline__ void add(float x) {
    const float t = hi + x;
    if (fabsf(hi) >= fabsf(x))
      lo += (hi - t) + x;
    else
      lo += (x - t) + hi;
    hi = t;
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// Sec. 1.4 energy correction in the state's precision class: double computes it in
// double; float computes the dense branch in double-float and the (rare) vacuum branch
// in double.  Returns 1 for the vacuum branch.
template <typename T>
__device__ __forceinline__ int correct_energy(T u[6], double rho_vac);
template <>
__device__ __forceinline__ int correct_energy<double>(double u[6], double rho_vac) {
  return energy_correction<false>(u, rho_vac);
}
// rho_vac_up = rho_vac rounded up to float: for any float x, x < rho_vac_up exactly when
// x < rho_vac (no float lies in [rho_vac, rho_vac_up) other than rho_vac itself).
// The two branches separately, for callers that batch cells: whether u takes the vacuum
// branch, the dense branch's rho eps, and the vacuum branch applied to u.
__device__ __forceinline__ bool vacuum_cell_f32(const float u[6], float rho_vac_up) {
  const float m2 = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
  return u[0] < rho_vac_up && m2 > 0.f;
}
__device__ __forceinline__ float dense_eps_f32(const float u[6]) {
  const float e = internal_energy_ff(u[0], u[1], u[2], u[3], u[4]);
  return e > 0.f ? e : u[5];
}
__device__ __forceinline__ void vacuum_correct_f32(float u[6], double rho_vac) {
  double d[6] = {u[0], u[1], u[2], u[3], u[4], u[5]};
  energy_correction<false>(d, rho_vac);
  u[1] = (float)d[1];
  u[2] = (float)d[2];
  u[3] = (float)d[3];
  u[5] = (float)d[5];
}
// The same two branches on a double-float state (low parts ul of rho, m, rho E): the dense
// value of rho eps, and the vacuum branch in double on hi + lo (m's pairs and rho eps
// rewritten).
__device__ __forceinline__ float dense_eps_df(const float u[6], const float ul[5]) {
  const float mh[3] = {u[1], u[2], u[3]}, ml[3] = {ul[1], ul[2], ul[3]};
  const float e = internal_energy_df(u[0], ul[0], mh, ml, u[4], ul[4]);
  return e > 0.f ? e : u[5];
}
// PLAIN: in the batch kernel, whose update pass is unrolled over four cells and would carry the
// shortcuts' code for a branch that is hardly taken (152 instances of 3000 cells, 16 steps: 348
// us with them, 343 without; the tile kernel is no faster without).
template <bool PLAIN>
__device__ __forceinline__ void vacuum_correct_df(float u[6], float ul[5], double rho_vac) {
  double d[6];
#pragma unroll
  for (int f = 0; f < 5; f++) d[f] = (double)u[f] + (double)ul[f];
  d[5] = u[5];
  energy_correction<PLAIN>(d, rho_vac);
#pragma unroll
  for (int a = 1; a <= 3; a++) df_split(d[a], u[a], ul[a]);
  u[5] = (float)d[5];
}
__device__ __forceinline__ int correct_energy_f32(float u[6], float rho_vac_up, double rho_vac) {
  if (vacuum_cell_f32(u, rho_vac_up)) {
    vacuum_correct_f32(u, rho_vac);
    return 1;
  }
  u[5] = dense_eps_f32(u);
  return 0;
}
template <>
__device__ __forceinline__ int correct_energy<float>(float u[6], double rho_vac) {
  return correct_energy_f32(u, __double2float_ru(rho_vac), rho_vac);
}

// Boundary handling by index mapping: interior coordinate read for coordinate c of an
// axis with n cells (outflow: clamp; periodic: wrap; reflecting: mirror, flip = 1; halo:
// the cell itself, stored up to kHaloCells beyond the face by the caller -- a neighbouring
// slab's cells).  Coordinates further than that outside the domain (only read for cells
// that produce no output) are clamped into range.
constexpr int kHaloCells = 3;
__device__ __forceinline__ int bc_map(int c, int n, int lo, int hi, int& flip) {
  flip = 0;
  if ((unsigned)c < (unsigned)n) return c;
  const int bc = c < 0 ? lo : hi;
  int r;
  if (bc == 1) {
    r = c < 0 ? c + n : c - n;
  } else if (bc == 2) {
    flip = 1;
    r = c < 0 ? -1 - c : 2 * n - 1 - c;
  } else if (bc == 3) {
    return c < 0 ? max(c, -kHaloCells) : min(c, n - 1 + kHaloCells);
  } else {
    r = c;
  }
  return min(max(r, 0), n - 1);
}

struct GridGeom {
  int n[3];
  int bc[6];
  long long nxy, ncell;
};

// Sign of field f (0..5; -1 for a scalar) at a cell reached through the mirrors in flips.
__device__ __forceinline__ bool field_flipped(int f, int flips) {
  return f >= 1 && f <= 3 && ((flips >> (f - 1)) & 1);
}

}  // namespace ppml
