// Shared pieces of the step kernels (Kulikov & Vorobyov, arXiv:1607.01105): kernel
// arguments, device-resident step scalars, deterministic per-CTA reductions of the CFL
// maxima (Sec. 1.1) and of the FP64 conservation sums, and the standalone
// diagnostics kernel.
#pragma once
#include "ppml_device.cuh"

namespace ppml {

constexpr int NT = 256;  // threads of the diagnostics kernel

struct Partial {
  double s[6];
  double vmax, cmax;
  unsigned long long nvac, nbad;
};

// Device-resident step scalars (one block per grid handle).
struct DevScalars {
  double t, dt, vmax, cmax, sums[6];
  long long steps, n_vac, n_bad;
  unsigned flags;
  unsigned arrived;  // CTAs of the running Lagrangian launch that have stored their partial
};

// What the partials of a state become: mode 0, the device scalars S of a state; 1, the same
// after a step; 2, the maxima, sums and counts in red[PPML_REDUCE_LEN] (a slab's share, for
// an all-reduce over the slabs).
struct Finalize {
  DevScalars* S;
  double* red;
  double cfl, hmin, vol, t_end;
  int mode;
};

template <typename T>
struct MarchArgs {
  const T* u[6];  // input fields
  T* out[6];      // output fields (out[0] NULL: rho is not written)
  // FP32 double-float states: low parts of rho, m_x, m_y, m_z, rho E of the input and the
  // output (all NULL for plain FP32 and FP64 states; outlo[0] NULL when out[0] is)
  const T* ulo[5];
  T* outlo[5];
  const T* phi;   // optional potential (Eulerian stage)
  GridGeom g;
  double h[3];
  double gamma;
  double dt_host;        // used when dt_dev == NULL
  const double* dt_dev;  // device-resident step
  double rho_vac;
  Partial* partials;      // per tile of the Lagrangian stage, at the tile's x-major index
  int tiles_x, tiles_y, tiles_z;  // tile grid of the stage kernels
  int tile_order;         // launch order of the tiles (TileOrder)
  int any_reflect;       // a reflecting wall exists (its sign flips need register copies)
  int flags;             // PPML_FIRST_ORDER, PPML_VHAT_1PT
  Finalize fin;          // of the Lagrangian stage's partials
  // FP32 with three active axes: the tiles' face velocities (ppml_tile_f32.cuh), room for
  // face_tiles tiles; a launch covers the blocks from tile_first on, and the array's first
  // tile is face_first (set by the launcher where the tiles take several launches)
  T* face;
  int face_tiles, tile_first, face_first;
  const T* inflow;       // [face][field]: the prescribed ghost states of inflow faces
  int any_inflow;        // an inflow face exists (selects the kernels that read them)
};

__device__ __forceinline__ double read_tau(const double* dt_dev, double dt_host) {
  return dt_dev ? *dt_dev : dt_host;
}

// The step size and tau / h per axis, formed by one thread of the CTA per axis (a division of
// a lone thread is ten dependent FP64 instructions of 76 cycles) and shared.  Contains a CTA
// barrier.
__device__ __forceinline__ void cta_step_constants(const double* dt_dev, double dt_host,
                                                   const double h[3], double out[4]) {
  __shared__ double s[4];
  if (threadIdx.x < 3) {
    const double tau = read_tau(dt_dev, dt_host);
    const double ha = threadIdx.x == 0 ? h[0] : (threadIdx.x == 1 ? h[1] : h[2]);
    if (threadIdx.x == 0) s[0] = tau;
    s[1 + threadIdx.x] = tau / ha;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; q++) out[q] = s[q];
}

// ------------------------------------------------------------------ block reduction

// The warps' shares folded in a fixed order into out[slot], a thread of the first warp per
// quantity (one thread folding all eight took 13 k cycles of 64 dependent FP64 operations at
// the end of every tile).  The stores are ordered before the warp's return.
template <int NW>
__device__ __forceinline__ void fold_warps(const double (*sh)[8], const unsigned long long (*shc)[2],
                                           Partial* out, int slot) {
  const int q = threadIdx.x;
  if (q < 6) {
    double v = 0.0;
#pragma unroll
    for (int w = 0; w < NW; w++) v = f64::plus(v, sh[w][q]);
    out[slot].s[q] = v;
  } else if (q < 8) {  // nonnegative: ordered as integers
    unsigned long long m = 0;
#pragma unroll
    for (int w = 0; w < NW; w++) m = max(m, (unsigned long long)__double_as_longlong(sh[w][q]));
    (q == 6 ? out[slot].vmax : out[slot].cmax) = __longlong_as_double((long long)m);
  } else if (q < 10) {
    unsigned long long n = 0;
#pragma unroll
    for (int w = 0; w < NW; w++) n += shc[w][q - 8];
    (q == 8 ? out[slot].nvac : out[slot].nbad) = n;
  }
}

// Writes the CTA's partial to out[slot].
template <int NTHREADS>
__device__ __forceinline__ void block_reduce_store(double s[6], double vmax, double cmax,
                                                   unsigned long long nvac,
                                                   unsigned long long nbad, Partial* out,
                                                   int slot) {
  __shared__ double sh[NTHREADS / 32][8];
  __shared__ unsigned long long shc[NTHREADS / 32][2];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int f = 0; f < 6; f++) s[f] = f64::plus(s[f], __shfl_down_sync(0xffffffffu, s[f], o));
    // nonnegative: ordered as integers
    vmax = __longlong_as_double(max(__double_as_longlong(vmax),
                                    __double_as_longlong(__shfl_down_sync(0xffffffffu, vmax, o))));
    cmax = __longlong_as_double(max(__double_as_longlong(cmax),
                                    __double_as_longlong(__shfl_down_sync(0xffffffffu, cmax, o))));
    nvac += __shfl_down_sync(0xffffffffu, nvac, o);
    nbad += __shfl_down_sync(0xffffffffu, nbad, o);
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    for (int f = 0; f < 6; f++) sh[w][f] = s[f];
    sh[w][6] = vmax;
    sh[w][7] = cmax;
    shc[w][0] = nvac;
    shc[w][1] = nbad;
  }
  __syncthreads();
  fold_warps<NTHREADS / 32>(sh, shc, out, slot);
}

// (hi, lo) += (bh, bl) in double-float (TwoSum of the high parts, then renormalised).
__device__ __forceinline__ void ff_add(float& hi, float& lo, float bh, float bl) {
  float s, e;
  two_sum(hi, bh, s, e);
  e += lo + bl;
  hi = s + e;
  lo = e - (hi - s);
}

// block_reduce_store for the FP32 stage kernels: the warp level of the sums runs in
// double-float (FP32 operations only), the maxima in float (exact) and the counters in
// 32 bits; warp leaders convert to double and fold_warps folds the warps in a fixed order.
template <int NTHREADS>
__device__ __forceinline__ void block_reduce_store_f32(const float hi_in[6], const float lo_in[6],
                                                       float vmax, float cmax, unsigned nvac,
                                                       unsigned nbad, Partial* out, int slot) {
  float hi[6], lo[6];
#pragma unroll
  for (int f = 0; f < 6; f++) {
    hi[f] = hi_in[f];
    lo[f] = lo_in[f];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int f = 0; f < 6; f++) {
      const float bh = __shfl_down_sync(0xffffffffu, hi[f], o);
      const float bl = __shfl_down_sync(0xffffffffu, lo[f], o);
      ff_add(hi[f], lo[f], bh, bl);
    }
    vmax = fmaxf(vmax, __shfl_down_sync(0xffffffffu, vmax, o));
    cmax = fmaxf(cmax, __shfl_down_sync(0xffffffffu, cmax, o));
    nvac += __shfl_down_sync(0xffffffffu, nvac, o);
    nbad += __shfl_down_sync(0xffffffffu, nbad, o);
  }
  __shared__ double sh[NTHREADS / 32][8];
  __shared__ unsigned long long shc[NTHREADS / 32][2];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    for (int f = 0; f < 6; f++) sh[w][f] = (double)hi[f] + (double)lo[f];
    sh[w][6] = vmax;
    sh[w][7] = cmax;
    shc[w][0] = nvac;
    shc[w][1] = nbad;
  }
  __syncthreads();
  fold_warps<NTHREADS / 32>(sh, shc, out, slot);
}

// The device scalars from the maxima, sums (times the cell volume) and counts of a state:
// advance: the state ends a step of tau (t += tau, clipped to t_end; steps + 1).  Then the
// next CFL step (Sec. 1.1) clipped to the remaining time, and the flags.
__device__ __forceinline__ void apply_scalars(DevScalars* S, double vmax, double cmax,
                                              const double* sums, double nvac, double nbad,
                                              int advance, double tau, double cfl, double hmin,
                                              double t_end) {
  double tn = S->t;
  if (advance) {
    tn = S->t + tau;
    if (t_end > 0.0 && tn > t_end) tn = t_end;
    S->t = tn;
    S->steps += 1;
    S->n_vac = (long long)nvac;
  }
  S->vmax = vmax;
  S->cmax = cmax;
  for (int f = 0; f < 6; f++) S->sums[f] = sums[f];
  S->n_bad = (long long)nbad;
  double dt = cfl * hmin / (vmax + cmax);
  if (t_end > 0.0 && dt > t_end - tn) dt = t_end - tn;
  if (!(dt > 0.0)) {
    dt = 0.0;
    S->flags |= 2u;  // PPML_FLAG_DT_ZERO
  }
  S->dt = dt;
  if (nbad > 0.0) S->flags |= 1u;  // PPML_FLAG_NONPHYSICAL
}

// Reduce nblk partials with one CTA of at least eight warps in an order that depends on nblk
// alone: a warp per sum (lane l takes partials l, l + 32, ..), one for the two maxima, one
// for the counts, so no FP64 lane idles (a tree over threads that each hold all eight values
// spent 12 us on 256 partials).  The partials may come from other CTAs of the same launch
// (read past L1).  tau: the step taken (mode 1).
__device__ __forceinline__ void finalize_cta(const Partial* P, int nblk, const Finalize& F,
                                             double tau) {
  __shared__ double res[8];
  __shared__ unsigned long long cnt[2];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int IN = 16;  // loads in flight per lane (the tail of the launch is their latency)
  if (w < 6) {
    double s = 0.0;
    for (int b0 = lane; b0 < nblk; b0 += 32 * IN) {
      double x[IN];
#pragma unroll
      for (int q = 0; q < IN; q++)
        x[q] = b0 + 32 * q < nblk ? __ldcg(&P[b0 + 32 * q].s[w]) : 0.0;
#pragma unroll
      for (int q = 0; q < IN; q++) s = f64::plus(s, x[q]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) res[w] = s * F.vol;
  } else if (w == 6) {  // maxima: nonnegative, so they order as integers
    unsigned long long v = 0, c = 0;
#pragma unroll 8
    for (int b = lane; b < nblk; b += 32) {
      v = max(v, (unsigned long long)__double_as_longlong(__ldcg(&P[b].vmax)));
      c = max(c, (unsigned long long)__double_as_longlong(__ldcg(&P[b].cmax)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      v = max(v, __shfl_down_sync(0xffffffffu, v, o));
      c = max(c, __shfl_down_sync(0xffffffffu, c, o));
    }
    if (lane == 0) {
      res[6] = __longlong_as_double((long long)v);
      res[7] = __longlong_as_double((long long)c);
    }
  } else if (w == 7) {
    unsigned long long nv = 0, nb = 0;
#pragma unroll 8
    for (int b = lane; b < nblk; b += 32) {
      nv += __ldcg(&P[b].nvac);
      nb += __ldcg(&P[b].nbad);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      nv += __shfl_down_sync(0xffffffffu, nv, o);
      nb += __shfl_down_sync(0xffffffffu, nb, o);
    }
    if (lane == 0) {
      cnt[0] = nv;
      cnt[1] = nb;
    }
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  if (F.mode == 2) {
    F.red[0] = res[6];
    F.red[1] = res[7];
    for (int f = 0; f < 6; f++) F.red[2 + f] = res[f];
    F.red[8] = (double)cnt[0];
    F.red[9] = (double)cnt[1];
    return;
  }
  apply_scalars(F.S, res[6], res[7], res, (double)cnt[0], (double)cnt[1], F.mode == 1, tau, F.cfl,
                F.hmin, F.t_end);
}

// End of a CTA of the Lagrangian stage whose first warp has stored its partial: the CTA that
// arrives last of nblk reduces them all.  The counter is zero between launches.
__device__ __forceinline__ void finalize_last(const Partial* P, int nblk, const Finalize& F,
                                              double tau) {
  __shared__ bool last;
  if (threadIdx.x < 32) {  // the partial's stores (fold_warps), visible before the arrival
    __threadfence();
    __syncwarp();
  }
  if (threadIdx.x == 0) {
    const unsigned n = atomicAdd(&F.S->arrived, 1u);
    last = n == (unsigned)nblk - 1u;
    if (last) {
      F.S->arrived = 0u;
      __threadfence();
    }
  }
  __syncthreads();
  if (last) finalize_cta(P, nblk, F, tau);
}

// Running per-thread sums of the six output fields: compensated float for the FP32
// path, plain double for the FP64 path.
template <typename T>
struct FieldSums;
template <>
struct FieldSums<float> {
  CompSum s[6];
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int f = 0; f < 6; f++) s[f].init();
  }
  __device__ __forceinline__ void add(const float u[6]) {
#pragma unroll
    for (int f = 0; f < 6; f++) s[f].add(u[f]);
  }
  // low parts of a double-float state's fields 0..4 (below the sums' rounding: plain adds)
  __device__ __forceinline__ void add_lo(const float lo[5]) {
#pragma unroll
    for (int f = 0; f < 5; f++) s[f].lo += lo[f];
  }
  __device__ __forceinline__ void get(double out[6]) const {
#pragma unroll
    for (int f = 0; f < 6; f++) out[f] = s[f].value();
  }
};
template <>
struct FieldSums<double> {
  double s[6];
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int f = 0; f < 6; f++) s[f] = 0.0;
  }
  __device__ __forceinline__ void add(const double u[6]) {
#pragma unroll
    for (int f = 0; f < 6; f++) s[f] = f64::plus(s[f], u[f]);
  }
  __device__ __forceinline__ void get(double out[6]) const {
#pragma unroll
    for (int f = 0; f < 6; f++) out[f] = s[f];
  }
};

// Per-cell part of the CFL step (Sec. 1.1) and of the non-physical check, in T.
template <typename T>
__device__ __forceinline__ void cell_speeds(const T u[6], T gamma, T gm1, T& vmax, T& cmax,
                                            unsigned long long& nbad) {
  const T rho = u[0];
  const T vx = u[1] / rho, vy = u[2] / rho, vz = u[3] / rho;
  const T v = sqrt(vx * vx + vy * vy + vz * vz);
  const T p = gm1 * u[5];
  const T c = sqrt(gamma * p / rho);
  bool ok = rho > T(0) && u[5] > T(0);
#pragma unroll
  for (int f = 0; f < 6; f++) ok = ok && isfinite(u[f]);
  if (ok) {
    vmax = fmax(vmax, v);
    cmax = fmax(cmax, c);
  } else {
    nbad++;
  }
}

// The CFL maxima of an FP64 tile without five divisions and roots per cell: every cell's
// speeds are bounded in float (RoughSpeeds: upper bounds), the largest lower bounds of the
// tile are taken, and only cells whose upper bound reaches them are evaluated exactly
// (ExactSpeeds, in cell_speeds' operations).  Values outside 2^-60 .. 2^60 have no float
// bound: their cells are always evaluated.
struct RoughSpeeds {
  float v, c;  // upper bounds; v = 0: at rest exactly; negative: not a physical cell
};
constexpr float kRoughUp = 1.00002f, kRoughDown = 0.99998f;  // truncations and approximations

__device__ __forceinline__ float truncated_float(double x) {  // x in float range or zero
  const unsigned h = (unsigned)f64::hi_word(x), l = (unsigned)f64::lo_word(x);
  if ((h << 1) == 0u) return 0.0f;
  return __uint_as_float((h & 0x80000000u) | (((h & 0x7fffffffu) - (896u << 20)) << 3) | (l >> 29));
}
__device__ __forceinline__ bool rough_range(double x) { return f64::exponent(x) - 963u <= 120u; }

__device__ __forceinline__ void rough_speeds(const double u[6], float ggm1, RoughSpeeds& r,
                                             float& vlow, float& clow,
                                             unsigned long long& nbad) {
  bool ok = f64::positive(u[0]) && f64::positive(u[5]);
#pragma unroll
  for (int f = 0; f < 6; f++) ok = ok && f64::finite(u[f]);
  if (!ok) {
    nbad++;
    r.v = r.c = -1.0f;
    return;
  }
  bool in = rough_range(u[0]) && rough_range(u[5]);
  bool rest = true;
#pragma unroll
  for (int f = 1; f <= 3; f++) {
    const bool z = f64::is_zero(u[f]);
    rest = rest && z;
    in = in && (z || rough_range(u[f]));
  }
  if (!in) {
    r.v = rest ? 0.0f : __int_as_float(0x7f800000);
    r.c = __int_as_float(0x7f800000);
    return;
  }
  const float ir = rcp_approx(truncated_float(u[0]));
  const float c = sqrt_approx(ggm1 * truncated_float(u[5]) * ir);
  float v = 0.0f;
  if (!rest) {
    const float mx = truncated_float(u[1]), my = truncated_float(u[2]), mz = truncated_float(u[3]);
    v = sqrt_approx(mx * mx + my * my + mz * mz) * ir;
  }
  r.v = v * kRoughUp;
  r.c = c * kRoughUp;
  vlow = fmaxf(vlow, v * kRoughDown);
  clow = fmaxf(clow, c * kRoughDown);
}

__device__ __forceinline__ float warp_max(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}

struct ExactSpeeds {
  double rho = 0.0, ei = 0.0;  // the last evaluated sound speed's cell (equal cells: equal speed)
  double last[4] = {0.0, 0.0, 0.0, 0.0};
  __device__ __forceinline__ void add(const double u[6], double gamma, double gm1, bool need_v,
                                      bool need_c, double& vmax, double& cmax) {
    if (need_v && !(f64::same_bits(u[0], last[0]) && f64::same_bits(u[1], last[1]) &&
                    f64::same_bits(u[2], last[2]) && f64::same_bits(u[3], last[3]))) {
#pragma unroll
      for (int f = 0; f < 4; f++) last[f] = u[f];
      const double vx = f64::over(u[1], u[0]), vy = f64::over(u[2], u[0]), vz = f64::over(u[3], u[0]);
      const double v = sqrt(vx * vx + vy * vy + vz * vz);
      vmax = fmax(vmax, v);
    }
    if (need_c && !(f64::same_bits(u[0], rho) && f64::same_bits(u[5], ei))) {
      rho = u[0];
      ei = u[5];
      const double p = gm1 * u[5];
      cmax = fmax(cmax, sqrt(gamma * p / u[0]));
    }
  }
};

// FP32 form for the stage kernels: one approximate reciprocal of rho, |v| = |m| / rho.
__device__ __forceinline__ void cell_speeds_f32(const float u[6], float gamma, float gm1,
                                                float& vmax, float& cmax,
                                                unsigned long long& nbad) {
  const float rho = u[0];
  const float ir = rcp_approx(rho);
  const float v = sqrt_approx(u[1] * u[1] + u[2] * u[2] + u[3] * u[3]) * ir;
  const float c = sqrt_approx(gamma * gm1 * u[5] * ir);
  bool ok = rho > 0.f && u[5] > 0.f;
#pragma unroll
  for (int f = 0; f < 6; f++) ok = ok && isfinite(u[f]);
  if (ok) {
    vmax = fmaxf(vmax, v);
    cmax = fmaxf(cmax, c);
  } else {
    nbad++;
  }
}

// ------------------------------------------------------------------ standalone diagnostics

template <typename T>
__global__ void __launch_bounds__(NT) diag_kernel(MarchArgs<T> A) {
  const long long n = A.g.ncell;
  FieldSums<T> sums;
  sums.init();
  T vmax = T(0), cmax = T(0);
  unsigned long long nbad = 0;
  const T gamma = T(A.gamma), gm1 = T(A.gamma - 1.0);
  for (long long idx = (long long)blockIdx.x * NT + threadIdx.x; idx < n;
       idx += (long long)gridDim.x * NT) {
    T u[6];
#pragma unroll
    for (int f = 0; f < 6; f++) u[f] = A.u[f][idx];
    sums.add(u);
    if constexpr (sizeof(T) == 4) {
      if (A.ulo[0]) {  // double-float state: the sums take the low parts too
        float lo[5];
#pragma unroll
        for (int f = 0; f < 5; f++) lo[f] = A.ulo[f][idx];
        sums.add_lo(lo);
      }
    }
    cell_speeds<T>(u, gamma, gm1, vmax, cmax, nbad);
  }
  double sd[6];
  sums.get(sd);
  block_reduce_store<NT>(sd, (double)vmax, (double)cmax, 0ull, nbad, A.partials, blockIdx.x);
}

}  // namespace ppml
