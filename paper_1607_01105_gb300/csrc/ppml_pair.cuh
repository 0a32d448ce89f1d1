// FP32 line pipelines of two quantities at a time (deviation form, ppml_device.cuh) on packed
// arithmetic: add, multiply and FMA of a register pair issue as one instruction (at the rate
// of two scalar ones), and whatever depends on the face alone is formed once for both.
#pragma once
#include "ppml_device.cuh"

namespace ppml {

// Two fields at once: packed additions, multiplications and FMAs (one issue slot for two).
__device__ __forceinline__ unsigned long long as_u64(float2 v) {
  return *reinterpret_cast<unsigned long long*>(&v);
}
__device__ __forceinline__ float2 as_f2(unsigned long long v) {
  return *reinterpret_cast<float2*>(&v);
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(as_u64(a)), "l"(as_u64(b)));
  return as_f2(r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(as_u64(a)), "l"(as_u64(b)));
  return as_f2(r);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(as_u64(a)), "l"(as_u64(b)), "l"(as_u64(c)));
  return as_f2(r);
}
__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, both(-1.0f), a); }

// Line pipeline of the deviation form for two quantities: push(q) takes the next position p;
// then q2 is the values and Pl, Pr the doubled deviations 2 (q0 - q^L), 2 (q^R - q0) of cell
// p - 2.  FLAT: the first-order variant (no deviations).
template <bool FLAT>
struct LinePair {
  float2 q2, q1, qn;  // values at p-2, p-1, p
  float2 d, s, l2;    // difference p-1 .. p, half slope and doubled left deviation of p-1
  float2 Pl, Pr;
  // half of the limited slope (Step 1): min(|l + r| / 4, |l|, |r|) with the differences'
  // common sign, 0 where their signs differ
  static __device__ __forceinline__ float2 half_slope(float2 l, float2 r) {
    const float2 c = mul2(add2(l, r), both(0.25f));
    return make_float2(min_xs(c.x, fmaxf(min_xs(l.x, r.x), 0.0f)),
                       min_xs(c.y, fmaxf(min_xs(l.y, r.y), 0.0f)));
  }
  __device__ __forceinline__ void start(float2 a, float2 b, float2 c) {
    q2 = a;
    q1 = b;
    qn = c;
    Pl = Pr = l2 = both(0.0f);
    d = sub2(c, b);
    s = half_slope(sub2(b, a), d);
  }
  __device__ __forceinline__ void push(float2 q) {
    if constexpr (!FLAT) {
      const float2 dn = sub2(q, qn);
      const float2 sn = half_slope(d, dn);
      // face between the two positions before q: doubled deviations d -+ (2/3)(sn - s)
      const float2 e = sub2(sn, s);
      const float2 r2 = fma2(e, both(-2.0f / 3.0f), d);
      const float2 t = make_float2(max_nan(min_xs_nan(l2.x, r2.x), 0.0f),
                                   max_nan(min_xs_nan(l2.y, r2.y), 0.0f));
      const float2 m = add2(t, t);
      Pl = make_float2(min_xs_nan(l2.x, m.x), min_xs_nan(l2.y, m.y));
      Pr = make_float2(min_xs_nan(r2.x, m.x), min_xs_nan(r2.y, m.y));
      l2 = fma2(e, both(2.0f / 3.0f), d);
      d = dn;
      s = sn;
    }
    q2 = q1;
    q1 = qn;
    qn = q;
  }
};

// th times the flux of eq. fluxonlagrangestage of two fields through a face, w = v^ th and
// c = dev_weights(|w|): w times the left cell's average when w >= 0, else the right cell's.
__device__ __forceinline__ float2 upwind_flux_pair(float w, const DevWeights& c, float2 ql, float2 Ll,
                                                   float2 Lr, float2 qr, float2 Rl, float2 Rr) {
  const bool left = w >= 0.0f;
  const float2 q = make_float2(left ? ql.x : qr.x, left ? ql.y : qr.y);
  const float2 x = make_float2(left ? Lr.x : -Rl.x, left ? Lr.y : -Rl.y);
  const float2 y = make_float2(left ? Ll.x : -Rr.x, left ? Ll.y : -Rr.y);
  return mul2(both(w), fma2(both(c.a), x, fma2(both(c.b), y, q)));
}
__device__ __forceinline__ float2 upwind_flux_pair(float w, float2 ql, float2 Ll, float2 Lr,
                                                   float2 qr, float2 Rl, float2 Rr) {
  return upwind_flux_pair(w, dev_weights(fabsf(w)), ql, Ll, Lr, qr, Rl, Rr);
}

// The acoustic face between a left and a right cell from the (v, p) pair of each (values q,
// doubled deviations L, R) and the cells' root weights: V and P of eqs. lowriemannvelocity /
// lowriemannpressure.
struct FaceCell {
  float2 q, L, R;    // (v, p) and its deviations
  float s, a, b;     // sqrt(rho), rho sqrt(rho), p sqrt(rho)
};
__device__ __forceinline__ void face_roots(FaceCell& c, float rho) {
  c.s = sqrt_approx(rho);
  c.a = rho * c.s;
  c.b = c.q.y * c.s;
}
__device__ __forceinline__ void acoustic_face(const FaceCell& l, const FaceCell& r, float gamma,
                                              float th, float& V, float& P) {
  const float A = l.a + r.a, lam = sqrt_approx(gamma * (l.b + r.b) * rcp_approx(A));
  const float Z = lam * A * rcp_approx(l.s + r.s);
  const DevWeights w = dev_weights(lam * th);
  const float2 right = fma2(both(w.a), l.R, fma2(both(w.b), l.L, l.q));
  const float2 left = fma2(both(-w.a), r.L, fma2(both(-w.b), r.R, r.q));
  const float2 sum = add2(right, left), dif = sub2(right, left);
  V = 0.5f * fmaf(dif.y, rcp_approx(Z), sum.x);
  P = 0.5f * fmaf(dif.x, Z, sum.y);
}

}  // namespace ppml
