// The stage kernels of grids with one or two active axes (plain float and double states).
//
// A 16^3 tile of such a grid holds 16 or 256 cells, and a thread that owns a line of it
// takes the six fields one after the other: the step is the latency of that chain (256 FP64
// cells in 1D: 1.18 ms a step; 256 x 256 in FP32: 119 us).  Here a CTA owns 16 x 16 cells
// (one axis: 32) with all fields in shared memory, and the work is spread over threads as
// (axis, line, segment of a line, field): a thread streams a few cells of one field (FP32:
// of two, packed), so the chain is short and both axes run at once.  A segment repeats six
// positions of start-up, which costs nothing on a machine that such a grid leaves idle.
// 256 x 256 in FP32: 28 us a step, 10 Eulerian, 18 Lagrangian.
// The line arithmetic is the tile kernels': FP64 the same bits.
#pragma once
#include "ppml_pair.cuh"
#include "ppml_tile.cuh"

namespace ppml {

constexpr int THIN_NT = 256;

// Cells of a CTA along the two axes and of a segment.  (FP64 grids of one axis have a pass per
// quantity in place of segments, below.)
template <typename T, bool TWO>
struct ThinShape {
  static constexpr int LA = TWO ? 16 : 32, LB = TWO ? 16 : 1;
  static constexpr int SEG = TWO ? 4 : 2;
  static constexpr int GB = TWO ? TH : 0;                  // ghosts along the second axis
  static constexpr int WA = LA + 2 * TH, WB = LB + 2 * GB;  // box
  static constexpr int PA = WA + 1;                        // box pitch
  static constexpr int BOX = PA * WB;
  static constexpr int CELLS = LA * LB;
  static constexpr int FACES = (LA + 1) * LB;               // of one axis (LA = LB if TWO)
};

// The active axes of the grid (B: -1 for one axis), the CTA's place, and the maps of its box.
struct ThinGeom {
  int axA, axB, a0, b0, tilesA, tilesB;
};
__host__ __device__ __forceinline__ ThinGeom thin_axes(const GridGeom& g) {
  ThinGeom t;
  t.axA = t.axB = -1;
  for (int q = 0; q < 3; q++) {
    if (g.n[q] == 1) continue;
    if (t.axA < 0)
      t.axA = q;
    else
      t.axB = q;
  }
  t.a0 = t.b0 = 0;
  t.tilesA = t.tilesB = 1;
  return t;
}
__host__ __device__ __forceinline__ bool thin_grid(const GridGeom& g) {
  const int act = (g.n[0] > 1) + (g.n[1] > 1) + (g.n[2] > 1);
  return (act == 1 || act == 2) && offsets_fit(g);
}
template <typename S>
__host__ __device__ __forceinline__ int thin_tiles(const GridGeom& g, ThinGeom& t) {
  t = thin_axes(g);
  t.tilesA = (g.n[t.axA] + S::LA - 1) / S::LA;
  t.tilesB = t.axB >= 0 ? (g.n[t.axB] + S::LB - 1) / S::LB : 1;
  return t.tilesA * t.tilesB;
}

struct ThinMaps {
  int off[2][38];
  int flip[2][38];
  int inflow[2][38];
};
template <typename S>
__device__ __forceinline__ void build_thin_maps(ThinMaps& M, const GridGeom& g, const ThinGeom& t) {
  for (int e = threadIdx.x; e < 2 * S::WA; e += THIN_NT) {
    const int q = e / S::WA, c = e % S::WA;
    const int ax = q == 0 ? t.axA : t.axB;
    if (ax < 0) continue;
    const int gc = (q == 0 ? t.a0 : t.b0) + c - TH, n = g.n[ax];
    int fl;
    const int m = bc_map(gc, n, g.bc[2 * ax], g.bc[2 * ax + 1], fl);
    M.off[q][c] = m * (ax == 0 ? 1 : (ax == 1 ? g.n[0] : (int)g.nxy));
    M.flip[q][c] = fl;
    M.inflow[q][c] = gc < 0 && g.bc[2 * ax] == PPML_BC_INFLOW
                         ? 2 * ax
                         : (gc >= n && g.bc[2 * ax + 1] == PPML_BC_INFLOW ? 2 * ax + 1 : -1);
  }
}
// Field f of the box through the maps (mirrored momenta negated, prescribed states at inflow
// faces, the later axis deciding).
template <typename T, typename S>
__device__ __forceinline__ void load_box(T* box, const MarchArgs<T>& A, int f, const ThinGeom& t,
                                         const ThinMaps& M) {
  for (int e = threadIdx.x; e < S::WA * S::WB; e += THIN_NT) {
    const int i = e % S::WA, j = e / S::WA;
    int o = M.off[0][i];
    bool neg = M.flip[0][i] && f == 1 + t.axA;
    int in = M.inflow[0][i];
    if (t.axB >= 0) {
      o += M.off[1][j];
      if (M.flip[1][j] && f == 1 + t.axB) neg = !neg;
      if (M.inflow[1][j] >= 0) in = M.inflow[1][j];
    }
    T v = __ldg(A.u[f] + o);
    if (neg) v = -v;
    if (in >= 0) v = __ldg(A.inflow + 6 * in + f);
    box[i + S::PA * j] = v;
  }
}

// A segment's task: axis q (0: A, 1: B), its first cell (i, j) of the tile, and its stride in
// the box.  Tasks: axis slowest, then segment, then line (consecutive threads take
// neighbouring lines).
template <typename S, int SEG>
struct ThinTask {
  int q, i, j, stride;
  __device__ __forceinline__ explicit ThinTask(int e) {
    constexpr int per = S::CELLS / SEG;  // of one axis
    q = e / per;
    const int r = e % per, line = r % S::LB, seg = r / S::LB;
    i = q == 0 ? SEG * seg : line;
    j = q == 0 ? line : SEG * seg;
    stride = q == 0 ? 1 : S::PA;
  }
  __device__ __forceinline__ int box() const { return (i + TH) + S::PA * (j + S::GB); }
  __device__ __forceinline__ int cell() const { return i + S::LA * j; }
  __device__ __forceinline__ int cell_stride() const { return q == 0 ? 1 : S::LA; }
};

// ------------------------------------------------------------------------- Eulerian stage

template <typename T, typename S>
struct ThinEulerSmem {
  T u[4][S::BOX];                  // rho, m_A, m_B, rho eps
  T dm[2][S::CELLS], dpv[2][S::CELLS], dv[2][S::CELLS];  // per axis
};

template <bool FLAT, int SEG, typename QF, typename EF>
__device__ __forceinline__ void thin_euler_line(QF q, float gamma, const AxisStep<float>& ks,
                                                EF emit) {
  float r[3] = {};  // rho of the last positions
  auto vp = [&](int p) {
    float rho, m, ei;
    q(p, rho, m, ei);
    r[0] = r[1];
    r[1] = r[2];
    r[2] = rho;
    return make_float2(m * rcp_approx(rho), ei);  // (ei: the pressure already)
  };
  LinePair<FLAT> ln;
  {
    const float2 a = vp(-3), b = vp(-2), c = vp(-1);
    ln.start(a, b, c);
  }
  ln.push(vp(0));
  ln.push(vp(1));
  FaceCell left{ln.q2, ln.Pl, ln.Pr};
  face_roots(left, r[0]);
  float Vp = 0.0f, Pp = 0.0f;
#pragma unroll
  for (int f = 0; f <= SEG; f++) {
    ln.push(vp(f + 2));
    FaceCell right{ln.q2, ln.Pl, ln.Pr};
    face_roots(right, r[0]);
    float V, P;
    acoustic_face(left, right, gamma, ks.th, V, P);
    if (f > 0) emit(f - 1, ks.th * (P - Pp), ks.th * (P * V - Pp * Vp), ks.th * (V - Vp));
    Vp = V;
    Pp = P;
    left = right;
  }
}

template <bool FLAT, int SEG, typename QF, typename EF>
__device__ __forceinline__ void thin_euler_line(QF q, double gamma, const AxisStep<double>& ks,
                                                EF emit) {
  double r[3] = {};
  auto push = [&](int p, double& v, double& pr) {
    double rho, m;
    q(p, rho, m, pr);
    r[0] = r[1];
    r[1] = r[2];
    r[2] = rho;
    v = f64::over(m, rho);
  };
  LineF64<FLAT> lv, lp;
  double v0, p0, v1, p1, v2, p2;
  push(-3, v0, p0);
  push(-2, v1, p1);
  push(-1, v2, p2);
  lv.start(v0, v1, v2);
  lp.start(p0, p1, p2);
#pragma unroll 1
  for (int p = 0; p < 2; p++) {
    push(p, v0, p0);
    lv.push(v0);
    lp.push(p0);
  }
  double vR = lv.R, vD = lv.D, vS = lv.S, pR = lp.R, pD = lp.D, pS = lp.S;
  RootWeights wl = root_weights(r[0], lp.q2);
  double Vp = 0.0, Pp = 0.0;
#pragma unroll 1
  for (int f = 0; f <= SEG; f++) {
    push(f + 2, v0, p0);
    lv.push(v0);
    lp.push(p0);
    const RootWeights wr = root_weights(r[0], lp.q2);
    double lam, Z, V, P;
    face_constants(wl, wr, gamma, lam, Z);
    wl = wr;
    const f64::Weights k = f64::weights(courant(lam, ks));
    riemann_vp(f64::average(true, vR, vD, vS, k), f64::average(false, lv.L, lv.D, lv.S, k),
               f64::average(true, pR, pD, pS, k), f64::average(false, lp.L, lp.D, lp.S, k), Z, V, P);
    if (f > 0)
      emit(f - 1, f64::times(ks.th, f64::diff(P, Pp)),
           f64::times(ks.th, f64::diff(f64::times(P, V), f64::times(Pp, Vp))),
           f64::times(ks.th, f64::diff(V, Vp)));
    Vp = V;
    Pp = P;
    vR = lv.R;
    vD = lv.D;
    vS = lv.S;
    pR = lp.R;
    pD = lp.D;
    pS = lp.S;
  }
}

template <typename T, bool FLAT, bool TWO>
__global__ void __launch_bounds__(THIN_NT) thin_eulerian(MarchArgs<T> A) {
  using S = ThinShape<T, TWO>;
  __shared__ ThinEulerSmem<T, S> M;
  __shared__ ThinMaps maps;
  __shared__ f64::Divisor hdiv[3];
  const GridGeom& g = A.g;
  ThinGeom t;
  thin_tiles<S>(g, t);
  t.a0 = (int)(blockIdx.x % t.tilesA) * S::LA;
  t.b0 = (int)(blockIdx.x / t.tilesA) * S::LB;
  build_thin_maps<S>(maps, g, t);
  if (sizeof(T) == 8 && threadIdx.x < 3) hdiv[threadIdx.x] = f64::divisor(A.h[threadIdx.x]);
  double stc[4];
  cta_step_constants(A.dt_dev, A.dt_host, A.h, stc);  // (a barrier)
  const T gamma = T(A.gamma), gm1 = T(A.gamma - 1.0);
  load_box<T, S>(M.u[0], A, 0, t, maps);
  load_box<T, S>(M.u[1], A, 1 + t.axA, t, maps);
  if (TWO) load_box<T, S>(M.u[2], A, 1 + t.axB, t, maps);
  load_box<T, S>(M.u[3], A, 5, t, maps);
  __syncthreads();
  constexpr int TASKS = (TWO ? 2 : 1) * S::CELLS / S::SEG;
  for (int e = threadIdx.x; e < TASKS; e += THIN_NT) {
    const ThinTask<S, S::SEG> k(e);
    const int ax = k.q == 0 ? t.axA : t.axB, b0 = k.box(), c0 = k.cell(), cs = k.cell_stride();
    const AxisStep<T> ks(stc[0], hdiv[ax], T(ax == 0 ? stc[1] : (ax == 1 ? stc[2] : stc[3])));
    const T* const r = M.u[0] + b0;
    const T* const m = M.u[1 + k.q] + b0;
    const T* const ei = M.u[3] + b0;
    thin_euler_line<FLAT, S::SEG>(
        [&](int p, T& rho, T& mv, T& pr) {
          const int o = p * k.stride;
          rho = r[o];
          mv = m[o];
          pr = gm1 * ei[o];
        },
        gamma, ks,
        [&](int c, T dm, T dpv, T dv) {
          M.dm[k.q][c0 + c * cs] = dm;
          M.dpv[k.q][c0 + c * cs] = dpv;
          M.dv[k.q][c0 + c * cs] = dv;
        });
  }
  __syncthreads();
  const int nxyz[3] = {1, g.n[0], (int)g.nxy};
  for (int c = threadIdx.x; c < S::CELLS; c += THIN_NT) {
    const int i = c % S::LA, j = c / S::LA;
    if (t.a0 + i >= g.n[t.axA] || (TWO && t.b0 + j >= g.n[t.axB])) continue;
    const int o = (t.a0 + i) * nxyz[t.axA] + (TWO ? (t.b0 + j) * nxyz[t.axB] : 0);
    const int b = (i + TH) + S::PA * (j + S::GB);
    T dpv = M.dpv[0][c], dv = M.dv[0][c];
    if (TWO) {
      dpv = add_term(dpv, M.dpv[1][c]);
      dv = add_term(dv, M.dv[1][c]);
    }
#pragma unroll
    for (int ax = 0; ax < 3; ax++) {
      if (ax == t.axA)
        A.out[1 + ax][o] = sub_term(M.u[1][b], M.dm[0][c]);
      else if (TWO && ax == t.axB)
        A.out[1 + ax][o] = sub_term(M.u[2][b], M.dm[1][c]);
      else
        A.out[1 + ax][o] = A.u[1 + ax][o];
    }
    A.out[4][o] = sub_term(A.u[4][o], dpv);
    A.out[5][o] = eps_update(M.u[3][b], gm1, dv);
    if (A.out[0]) A.out[0][o] = M.u[0][b];
  }
}

// ----------------------------------------------------------------------- Lagrangian stage

// What a face carries to the sweeps: FP32 the Courant velocity w = v^ tau/h; FP64 v^ and the
// weights of the characteristic averages.
template <typename T>
struct ThinFace;
template <>
struct ThinFace<float> {
  float w;
};
template <>
struct ThinFace<double> {
  double v;
  f64::Weights k;
};

template <typename T, typename S>
struct ThinLagSmem {
  T u[6][S::BOX];
  T v[2][S::BOX], sq[S::BOX];  // v_A, v_B and sqrt(rho) on the cells -1 .. L
  ThinFace<T> face[2][S::FACES];
  T d[2][6][S::CELLS];  // th (F+ - F-) per axis and field
};

// The template velocity (eq. veltemplate) of component axis at a box cell; sb, sc: box strides
// of the two other axes in the order of the formula (0: inactive, the cell itself).
template <typename T>
__device__ __forceinline__ T thin_template(const T* v, int o, int sb, int sc, bool one_point) {
  if (one_point) return v[o];
  if constexpr (sizeof(T) == 4) {
    const T corners = (v[o + sb + sc] + v[o + sb - sc]) + (v[o - sb + sc] + v[o - sb - sc]);
    const T edges = (v[o + sb] + v[o - sb]) + (v[o + sc] + v[o - sc]);
    return 0.0625f * corners + 0.125f * edges + 0.25f * v[o];
  } else {
    const T c0 = v[o + sb + sc], c1 = v[o + sb - sc], c2 = v[o - sb + sc], c3 = v[o - sb - sc];
    const T e0 = v[o + sb], e1 = v[o - sb], e2 = v[o + sc], e3 = v[o - sc];
    return f64::scale<-4>(c0 + c1 + c2 + c3) + f64::scale<-3>(e0 + e1 + e2 + e3) +
           f64::scale<-2>(v[o]);
  }
}

__device__ __forceinline__ ThinFace<float> thin_face(float pl, float pr, float sl, float sr,
                                                     const AxisStep<float>& ks) {
  return {(pr + pl) * rcp_approx(sr + sl) * ks.th};
}
__device__ __forceinline__ ThinFace<double> thin_face(double pl, double pr, double sl, double sr,
                                                      const AxisStep<double>& ks) {
  ThinFace<double> f;
  f.v = (pr + pl) / (sr + sl);
  f.k = f64::weights(courant(tabs(f.v), ks));
  return f;
}

// A segment of one line: FP32 two fields at once (f, f + 1), FP64 one.
template <bool FLAT, int SEG>
__device__ __forceinline__ void thin_lag_line(const float* u0, const float* u1, int stride,
                                              const ThinFace<float>* face, int fstride, float* d0,
                                              float* d1, int cs, float) {
  auto q = [&](int p) { return make_float2(u0[p * stride], u1[p * stride]); };
  LinePair<FLAT> ln;
  ln.start(q(-3), q(-2), q(-1));
  ln.push(q(0));
  ln.push(q(1));
  float2 ql = ln.q2, Ll = ln.Pl, Lr = ln.Pr, Fp = both(0.0f);
#pragma unroll
  for (int f = 0; f <= SEG; f++) {
    ln.push(q(f + 2));
    const float2 F = upwind_flux_pair(face[f * fstride].w, ql, Ll, Lr, ln.q2, ln.Pl, ln.Pr);
    if (f > 0) {
      const float2 d = sub2(F, Fp);
      d0[(f - 1) * cs] = d.x;
      d1[(f - 1) * cs] = d.y;
    }
    Fp = F;
    ql = ln.q2;
    Ll = ln.Pl;
    Lr = ln.Pr;
  }
}
template <bool FLAT, int SEG>
__device__ __forceinline__ void thin_lag_line(const double* u, const double*, int stride,
                                              const ThinFace<double>* face, int fstride, double* d,
                                              double*, int cs, double th) {
  LineF64<FLAT> ln;
  ln.start(u[-3 * stride], u[-2 * stride], u[-stride]);
  ln.push(u[0]);
  ln.push(u[stride]);
  double Rl = ln.R, Dl = ln.D, Sl = ln.S, Fp = 0.0;
#pragma unroll 1
  for (int f = 0; f <= SEG; f++) {
    ln.push(u[(f + 2) * stride]);
    const ThinFace<double> k = face[f * fstride];
    const bool left = f64::hi_word(k.v) >= 0;
    const double st =
        f64::average(left, left ? Rl : ln.L, left ? Dl : ln.D, left ? Sl : ln.S, k.k);
    const double F = f64::is_zero(k.v) && f64::finite(st) ? 0.0 : f64::plain_mul(k.v, st);
    if (f > 0) d[(f - 1) * cs] = f64::times(th, f64::diff(F, Fp));
    Fp = F;
    Rl = ln.R;
    Dl = ln.D;
    Sl = ln.S;
  }
}

template <typename T, bool FLAT, bool TWO>
__global__ void __launch_bounds__(THIN_NT) thin_lagrangian(MarchArgs<T> A) {
  using S = ThinShape<T, TWO>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ThinLagSmem<T, S>& M = *reinterpret_cast<ThinLagSmem<T, S>*>(smem_raw);
  __shared__ ThinMaps maps;
  __shared__ f64::Divisor hdiv[3];
  const GridGeom& g = A.g;
  ThinGeom t;
  const int tiles = thin_tiles<S>(g, t);
  t.a0 = (int)(blockIdx.x % t.tilesA) * S::LA;
  t.b0 = (int)(blockIdx.x / t.tilesA) * S::LB;
  build_thin_maps<S>(maps, g, t);
  if (sizeof(T) == 8 && threadIdx.x < 3) hdiv[threadIdx.x] = f64::divisor(A.h[threadIdx.x]);
  double stc[4];
  cta_step_constants(A.dt_dev, A.dt_host, A.h, stc);  // (a barrier)
  const T gamma = T(A.gamma), gm1 = T(A.gamma - 1.0);
  const bool one_point = (A.flags & PPML_VHAT_1PT) != 0;
  auto axis_step = [&](int ax) {
    return AxisStep<T>(stc[0], hdiv[ax], T(ax == 0 ? stc[1] : (ax == 1 ? stc[2] : stc[3])));
  };
#pragma unroll 1
  for (int f = 0; f < 6; f++) load_box<T, S>(M.u[f], A, f, t, maps);
  __syncthreads();
  // velocities and Roe weights on the cells -1 .. L
  constexpr int VA = S::LA + 2, VB = TWO ? S::LB + 2 : 1;
  for (int e = threadIdx.x; e < VA * VB; e += THIN_NT) {
    const int o = (e % VA + TH - 1) + S::PA * (e / VA + (TWO ? S::GB - 1 : 0));
    const T r = M.u[0][o];
    const T mA = t.axA == 0 ? M.u[1][o] : (t.axA == 1 ? M.u[2][o] : M.u[3][o]);
    const T mB = TWO ? (t.axB == 1 ? M.u[2][o] : M.u[3][o]) : T(0);
    if constexpr (sizeof(T) == 4) {
      const float ir = rcp_approx(r);
      M.v[0][o] = mA * ir;
      if (TWO) M.v[1][o] = mB * ir;
      M.sq[o] = sqrt_approx(r);
    } else {
      M.v[0][o] = f64::over(mA, r);
      if (TWO) M.v[1][o] = f64::over(mB, r);
      M.sq[o] = sqrt(r);
    }
  }
  __syncthreads();
  // face velocities: face f of line l of axis q at index f LB + l (axis B: f LA + l)
  for (int e = threadIdx.x; e < (TWO ? 2 : 1) * S::FACES; e += THIN_NT) {
    const int q = e / S::FACES, r = e % S::FACES, l = r % S::LB, f = r / S::LB;
    const int ax = q == 0 ? t.axA : t.axB;
    auto box_stride = [&](int axis) { return axis == t.axA ? 1 : (axis == t.axB ? S::PA : 0); };
    const int sb = box_stride((ax + 1) % 3), sc = box_stride((ax + 2) % 3);
    const int o = q == 0 ? (f + TH) + S::PA * (l + S::GB) : (l + TH) + S::PA * (f + S::GB);
    const int ol = o - (q == 0 ? 1 : S::PA);
    const T sl = M.sq[ol], sr = M.sq[o];
    const T pl = thin_template(M.v[q], ol, sb, sc, one_point) * sl;
    const T pr = thin_template(M.v[q], o, sb, sc, one_point) * sr;
    M.face[q][f * S::LB + l] = thin_face(pl, pr, sl, sr, axis_step(ax));
  }
  __syncthreads();
  constexpr int GROUP = sizeof(T) == 4 ? 2 : 1;  // fields of a task
  constexpr int SEGS = (TWO ? 2 : 1) * S::CELLS / S::SEG;
  for (int e = threadIdx.x; e < SEGS * (6 / GROUP); e += THIN_NT) {
    const ThinTask<S, S::SEG> k(e % SEGS);
    const int f = e / SEGS * GROUP;
    const int first = k.q == 0 ? k.i : k.j, line = k.q == 0 ? k.j : k.i;
    const int ax = k.q == 0 ? t.axA : t.axB;
    thin_lag_line<FLAT, S::SEG>(
        M.u[f] + k.box(), M.u[f + GROUP - 1] + k.box(), k.stride,
        &M.face[k.q][first * S::LB + line], S::LB, &M.d[k.q][f][k.cell()],
        &M.d[k.q][f + GROUP - 1][k.cell()], k.cell_stride(),
        T(ax == 0 ? stc[1] : (ax == 1 ? stc[2] : stc[3])));
  }
  __syncthreads();
  // updates, energy correction (Sec. 1.4), CFL maxima and sums
  FieldSums<T> sums;
  sums.init();
  T vmax = T(0), cmax = T(0);
  unsigned long long nvac = 0, nbad = 0;
  RoughSpeeds rough = {-1.0f, -1.0f};
  float vlow = 0.0f, clow = 0.0f;
  T u[6];
  const int nxyz[3] = {1, g.n[0], (int)g.nxy};
  static_assert(S::CELLS <= THIN_NT, "a cell per thread");
  {
    const int c = threadIdx.x, i = c % S::LA, j = c / S::LA;
    if (c < S::CELLS && t.a0 + i < g.n[t.axA] && (!TWO || t.b0 + j < g.n[t.axB])) {
      const int o = (t.a0 + i) * nxyz[t.axA] + (TWO ? (t.b0 + j) * nxyz[t.axB] : 0);
      const int b = (i + TH) + S::PA * (j + S::GB);
#pragma unroll
      for (int f = 0; f < 6; f++) {
        T d = M.d[0][f][c];
        if (TWO) d = add_term(d, M.d[1][f][c]);
        u[f] = sub_term(M.u[f][b], d);
      }
      nvac = correct_energy<T>(u, A.rho_vac);
#pragma unroll
      for (int f = 0; f < 6; f++) A.out[f][o] = u[f];
      sums.add(u);
      if constexpr (sizeof(T) == 4)
        cell_speeds_f32(u, gamma, gm1, vmax, cmax, nbad);
      else
        rough_speeds(u, (float)A.gamma * (float)(A.gamma - 1.0), rough, vlow, clow, nbad);
    }
  }
  if constexpr (sizeof(T) == 4) {
    float hi[6], lo[6];
#pragma unroll
    for (int f = 0; f < 6; f++) {
      hi[f] = sums.s[f].hi;
      lo[f] = sums.s[f].lo;
    }
    block_reduce_store_f32<THIN_NT>(hi, lo, vmax, cmax, (unsigned)nvac, (unsigned)nbad, A.partials,
                                    blockIdx.x);
  } else {
    __shared__ float low[THIN_NT / 32][2];
    vlow = warp_max(vlow);
    clow = warp_max(clow);
    if ((threadIdx.x & 31) == 0) {
      low[threadIdx.x >> 5][0] = vlow;
      low[threadIdx.x >> 5][1] = clow;
    }
    __syncthreads();
    for (int q = 0; q < THIN_NT / 32; q++) {
      vlow = fmaxf(vlow, low[q][0]);
      clow = fmaxf(clow, low[q][1]);
    }
    const bool nv = rough.v > 0.0f && rough.v >= vlow, nc = rough.c >= clow;
    if (nv || nc) {
      ExactSpeeds ex;
      ex.add(u, gamma, gm1, nv, nc, vmax, cmax);
    }
    double sd[6];
    sums.get(sd);
    block_reduce_store<THIN_NT>(sd, (double)vmax, (double)cmax, nvac, nbad, A.partials, blockIdx.x);
  }
  finalize_last(A.partials, tiles, A.fin, stc[0]);
}

// ------------------------------------------------- FP64 grids with one active axis
// One FP64 instruction of a lone warp takes 76 cycles, so even one cell's chain through a
// line segment (seven positions of start-up for two quantities, two faces of 75 instructions)
// is 25 us.  Here every quantity of the stage has its own pass over the CTA's 32 cells and
// their ghosts, spread over (quantity, cell): the chain is one slope, one face, one parabola,
// one face solve and one update (256 cells: 61 us a step with segments of one cell,
// 35 like this).

struct Thin1dEuler {
  static constexpr int L = 32, W = L + 2 * TH;  // positions -3 .. L+2 at index p + 3
  double r[W], m[W], ei[W];
  double q[2][W];             // v, p
  RootWeights w[W];           // of the cells -1 .. L
  double s[2][W], f[2][W];    // slopes; face p: between p-1 and p
  double PL[2][W], PR[2][W], D[2][W], S[2][W];
  double V[W], P[W];          // faces 0 .. L
};

template <bool FLAT>
__global__ void __launch_bounds__(THIN_NT) thin1d_eulerian_f64(MarchArgs<double> A) {
  using E = Thin1dEuler;
  using S1 = ThinShape<double, false>;
  static_assert(E::L == S1::LA, "cells of a CTA");
  __shared__ E M;
  __shared__ ThinMaps maps;
  __shared__ f64::Divisor hdiv[3];
  const GridGeom& g = A.g;
  ThinGeom t;
  thin_tiles<S1>(g, t);
  t.a0 = (int)blockIdx.x * E::L;
  build_thin_maps<S1>(maps, g, t);
  if (threadIdx.x < 3) hdiv[threadIdx.x] = f64::divisor(A.h[threadIdx.x]);
  double stc[4];
  cta_step_constants(A.dt_dev, A.dt_host, A.h, stc);  // (a barrier)
  const double gamma = A.gamma, gm1 = A.gamma - 1.0;
  const int ax = t.axA, tid = threadIdx.x;
  const AxisStep<double> ks(stc[0], hdiv[ax], stc[1 + ax]);
  load_box<double, S1>(M.r, A, 0, t, maps);
  load_box<double, S1>(M.m, A, 1 + ax, t, maps);
  load_box<double, S1>(M.ei, A, 5, t, maps);
  __syncthreads();
  // v, p, root weights: 64 tasks per quantity, one warp pair each
  const int job = tid / 64, c = tid % 64;
  if (c < E::W) {
    if (job == 0) M.q[0][c] = f64::over(M.m[c], M.r[c]);
    if (job == 1) M.q[1][c] = f64::plain_mul(gm1, M.ei[c]);
    if (job == 2 && c >= 2 && c < E::W - 2)
      M.w[c] = root_weights(M.r[c], f64::plain_mul(gm1, M.ei[c]));
  }
  __syncthreads();
  if (job < 2) {
    double* const q = M.q[job];
    // slopes of the cells -2 .. L+1
    if (c >= 1 && c < E::W - 1)
      M.s[job][c] = FLAT ? 0.0
                         : f64::slope(f64::diff(q[c], q[c - 1]), f64::diff(q[c + 1], q[c]), q[c - 1],
                                      q[c + 1]);
  }
  __syncthreads();
  if (job < 2 && c >= 2 && c < E::W - 1)  // faces -1 .. L+1
    M.f[job][c] = f64::face(M.q[job][c - 1], M.q[job][c], M.s[job][c - 1], M.s[job][c]);
  __syncthreads();
  if (job < 2 && c >= 2 && c < E::W - 2) {  // cells -1 .. L
    const double q0 = M.q[job][c];
    double Lf = M.f[job][c], Rf = M.f[job][c + 1], D = 0.0, S = 0.0;
    if (FLAT)
      Lf = Rf = q0;
    else
      f64::parabola(q0, Lf, Rf, D, S);
    M.PL[job][c] = Lf;
    M.PR[job][c] = Rf;
    M.D[job][c] = D;
    M.S[job][c] = S;
  }
  __syncthreads();
  if (job == 0 && c >= TH && c <= TH + E::L) {  // face c - 3, between cells c-1 and c
    double lam, Z;
    face_constants(M.w[c - 1], M.w[c], gamma, lam, Z);
    const f64::Weights k = f64::weights(courant(lam, ks));
    riemann_vp(f64::average(true, M.PR[0][c - 1], M.D[0][c - 1], M.S[0][c - 1], k),
               f64::average(false, M.PL[0][c], M.D[0][c], M.S[0][c], k),
               f64::average(true, M.PR[1][c - 1], M.D[1][c - 1], M.S[1][c - 1], k),
               f64::average(false, M.PL[1][c], M.D[1][c], M.S[1][c], k), Z, M.V[c], M.P[c]);
  }
  __syncthreads();
  // updates: a thread per field and cell; cell i at index b
  const int i = c, b = c + TH;
  if (i < E::L && t.a0 + i < g.n[ax]) {
    const long long o = t.a0 + i;  // (the only active axis: contiguous)
    const double Vm = M.V[b], Vp = M.V[b + 1], Pm = M.P[b], Pp = M.P[b + 1];
    if (job == 0) {
#pragma unroll
      for (int q = 0; q < 3; q++)
        A.out[1 + q][o] = q == ax ? f64::minus(M.m[b], f64::times(ks.th, f64::diff(Pp, Pm)))
                                  : A.u[1 + q][o];
    } else if (job == 1) {
      const double d = f64::diff(f64::times(Pp, Vp), f64::times(Pm, Vm));
      A.out[4][o] = f64::minus(A.u[4][o], f64::times(ks.th, d));
    } else if (job == 2) {
      A.out[5][o] = eps_update(M.ei[b], gm1, f64::times(ks.th, f64::diff(Vp, Vm)));
      if (A.out[0]) A.out[0][o] = M.r[b];
    }
  }
}

struct Thin1dLag {
  static constexpr int L = 32, W = L + 2 * TH;
  double u[6][W + 1];
  double pr[W], sq[W];        // v sqrt(rho), sqrt(rho) of the cells -1 .. L
  double v[W];                // v^ of the faces 0 .. L
  f64::Weights k[W];
  double s[6][W], f[6][W], PL[6][W], PR[6][W], D[6][W], S[6][W];
  double F[6][W];
  double n[6][L];             // the updated cells
};

template <bool FLAT>
__global__ void __launch_bounds__(THIN_NT) thin1d_lagrangian_f64(MarchArgs<double> A) {
  using E = Thin1dLag;
  using S1 = ThinShape<double, false>;
  __shared__ E M;
  __shared__ ThinMaps maps;
  __shared__ f64::Divisor hdiv[3];
  const GridGeom& g = A.g;
  ThinGeom t;
  const int tiles = thin_tiles<S1>(g, t);
  t.a0 = (int)blockIdx.x * E::L;
  build_thin_maps<S1>(maps, g, t);
  if (threadIdx.x < 3) hdiv[threadIdx.x] = f64::divisor(A.h[threadIdx.x]);
  double stc[4];
  cta_step_constants(A.dt_dev, A.dt_host, A.h, stc);  // (a barrier)
  const double gamma = A.gamma, gm1 = A.gamma - 1.0;
  const int ax = t.axA, tid = threadIdx.x;
  const AxisStep<double> ks(stc[0], hdiv[ax], stc[1 + ax]);
  const bool one_point = (A.flags & PPML_VHAT_1PT) != 0;
#pragma unroll 1
  for (int f = 0; f < 6; f++) load_box<double, S1>(M.u[f], A, f, t, maps);
  __syncthreads();
  // slopes of the fields (38 threads each), and beside them the velocities and Roe weights
  // of the cells -1 .. L (the template of a cell whose transverse neighbours are itself)
  for (int e = tid; e < 6 * E::W; e += THIN_NT) {
    const int f = e / E::W, c = e % E::W;
    const double* const q = M.u[f];
    if (c >= 1 && c < E::W - 1)
      M.s[f][c] = FLAT ? 0.0
                       : f64::slope(f64::diff(q[c], q[c - 1]), f64::diff(q[c + 1], q[c]),
                                    q[c - 1], q[c + 1]);
  }
  if (tid >= THIN_NT - 64 && tid - (THIN_NT - 64) < E::L + 2) {
    const int c = tid - (THIN_NT - 64) + 2;
    const double r = M.u[0][c], sq = sqrt(r);
    const double v = f64::over(ax == 0 ? M.u[1][c] : (ax == 1 ? M.u[2][c] : M.u[3][c]), r);
    // corners and edges of eq. veltemplate along an axis with its transverse ones inactive
    const double four = v + v + v + v;
    const double vt = one_point ? v
                                : f64::scale<-4>(four) + f64::scale<-3>(four) + f64::scale<-2>(v);
    M.sq[c] = sq;
    M.pr[c] = vt * sq;
  }
  __syncthreads();
  for (int e = tid; e < 6 * E::W; e += THIN_NT) {
    const int f = e / E::W, c = e % E::W;
    if (c >= 2 && c < E::W - 1)
      M.f[f][c] = f64::face(M.u[f][c - 1], M.u[f][c], M.s[f][c - 1], M.s[f][c]);
  }
  if (tid >= THIN_NT - 64 && tid - (THIN_NT - 64) <= E::L) {
    const int c = tid - (THIN_NT - 64) + TH;  // face c - 3
    const ThinFace<double> w = thin_face(M.pr[c - 1], M.pr[c], M.sq[c - 1], M.sq[c], ks);
    M.v[c] = w.v;
    M.k[c] = w.k;
  }
  __syncthreads();
  for (int e = tid; e < 6 * E::W; e += THIN_NT) {
    const int f = e / E::W, c = e % E::W;
    if (c < 2 || c >= E::W - 2) continue;
    const double q0 = M.u[f][c];
    double Lf = M.f[f][c], Rf = M.f[f][c + 1], D = 0.0, S = 0.0;
    if (FLAT)
      Lf = Rf = q0;
    else
      f64::parabola(q0, Lf, Rf, D, S);
    M.PL[f][c] = Lf;
    M.PR[f][c] = Rf;
    M.D[f][c] = D;
    M.S[f][c] = S;
  }
  __syncthreads();
  for (int e = tid; e < 6 * (E::L + 1); e += THIN_NT) {
    const int f = e / (E::L + 1), c = e % (E::L + 1) + TH;
    const double v = M.v[c];
    const bool left = f64::hi_word(v) >= 0;
    const int o = left ? c - 1 : c;
    const double st = f64::average(left, left ? M.PR[f][o] : M.PL[f][o], M.D[f][o], M.S[f][o], M.k[c]);
    M.F[f][c] = f64::is_zero(v) && f64::finite(st) ? 0.0 : f64::plain_mul(v, st);
  }
  __syncthreads();
  for (int e = tid; e < 6 * E::L; e += THIN_NT) {
    const int f = e / E::L, i = e % E::L, b = i + TH;
    M.n[f][i] = f64::minus(M.u[f][b], f64::times(ks.th, f64::diff(M.F[f][b + 1], M.F[f][b])));
  }
  __syncthreads();
  // a cell per thread of the first warp: energy correction, CFL maxima; sums over the warp
  FieldSums<double> sums;
  sums.init();
  double vmax = 0.0, cmax = 0.0;
  unsigned long long nvac = 0, nbad = 0;
  static_assert(E::L == 32, "the cells are one warp's");
  if (tid < 32) {
    double u[6];
    RoughSpeeds rough = {-1.0f, -1.0f};
    float vlow = 0.0f, clow = 0.0f;
    if (t.a0 + tid < g.n[ax]) {
      const long long o = t.a0 + tid;
#pragma unroll
      for (int f = 0; f < 6; f++) u[f] = M.n[f][tid];
      nvac = correct_energy<double>(u, A.rho_vac);
#pragma unroll
      for (int f = 0; f < 6; f++) A.out[f][o] = u[f];
      sums.add(u);
      rough_speeds(u, (float)A.gamma * (float)(A.gamma - 1.0), rough, vlow, clow, nbad);
    }
    vlow = warp_max(vlow);
    clow = warp_max(clow);
    const bool nv = rough.v > 0.0f && rough.v >= vlow, nc = rough.c >= clow;
    if (nv || nc) {
      ExactSpeeds ex;
      ex.add(u, gamma, gm1, nv, nc, vmax, cmax);
    }
  }
  double sd[6];
  sums.get(sd);
  block_reduce_store<THIN_NT>(sd, vmax, cmax, nvac, nbad, A.partials, blockIdx.x);
  finalize_last(A.partials, tiles, A.fin, stc[0]);
}

}  // namespace ppml
