// FP32 stages of grids with three active axes (plain float states), 16^3 tiles:
//
//   eulerian_sweep_f32  the Eulerian stage (Sec. 1.1/1.2), with the gravity source terms
//
// and the Lagrangian stage in two kernels:
//
//   face_velocity_f32   eqs. veltemplate and modspaceaveragevelocitylagrange: the Courant
//                       velocities w = v^ tau/h of every face of every 16^3 tile, into a
//                       scratch array in the order the sweeps read it
//   lagrangian_sweep_f32  eqs. fluxonlagrangestage, genlagrange, the energy consistency of
//                       Sec. 1.4, the CFL maxima and sums
//
// Why two: one kernel that holds the velocity boxes, the face velocities of its lines, a
// field with its halos and an accumulator fills 105 KB of shared memory and waits for staging
// with nothing beside it (issue slots 52 % busy).  With the velocities coming from L2 in
// coalesced rows the weights of a face are formed once for two fields, and no staging phase is
// left: the z sweep reads its columns from global memory itself, a few positions ahead, and
// leaves them in shared memory (70 KB for two fields) for the x and y sweeps.
//
// Bound by instruction issue (about half of the slots busy) and the ALU pipe that the minima
// and selects share, with two CTAs of eight warps an SM: the shared memory would hold three,
// the 128 registers a thread do not (at 80: 2844 us for two 256^3 steps against 2685).  256^3, one step, before and after: Eulerian
// 580 -> 315 us, Lagrangian 1325 -> 592 + 166 us; DRAM traffic 41.7 B/cell, 26.5 + 65.7.
#pragma once
#include "ppml_pair.cuh"
#include "ppml_tile.cuh"

namespace ppml {

// Face velocities of a tile: [axis][face 0..16][line], line a + 16 b of that axis.
constexpr int FACE_AXIS = (TB + 1) * TN;
constexpr int FACE_TILE = 3 * FACE_AXIS;

// Tile maps with 32-bit offsets (a grid has fewer than 2^31 cells), as TileMaps.
struct TileMaps32 {
  int off[3][TW];
  int flip[3][TW];    // the axis is mirrored there
  int inflow[3][TW];  // the inflow face whose ghost region the coordinate lies in, or -1
};
__device__ __forceinline__ void build_maps32(TileMaps32& M, const GridGeom& g, const TileGeom& t) {
  for (int e = threadIdx.x; e < 3 * TW; e += blockDim.x) {
    const int ax = e / TW, c = e % TW - TH;
    const int o = ax == 0 ? t.i0 : (ax == 1 ? t.j0 : t.k0);
    const int gc = o + c, n = g.n[ax];
    int fl;
    const int m = bc_map(gc, n, g.bc[2 * ax], g.bc[2 * ax + 1], fl);
    M.off[ax][c + TH] = m * (ax == 0 ? 1 : (ax == 1 ? g.n[0] : (int)g.nxy));
    M.flip[ax][c + TH] = fl;
    M.inflow[ax][c + TH] = gc < 0 && g.bc[2 * ax] == PPML_BC_INFLOW
                               ? 2 * ax
                               : (gc >= n && g.bc[2 * ax + 1] == PPML_BC_INFLOW ? 2 * ax + 1 : -1);
  }
}

// ------------------------------------------------------------------------ face velocities

constexpr int FV_W = TB + 2;                 // columns -1..16 along x and y
constexpr int FV_THREADS = 352;              // 18 x 18 columns in eleven warps
constexpr int FV_PLANE = FV_W * FV_W;

// A CTA marches the planes k = -1..16 of its tile; thread (i, j) owns a column.  The 9-point
// template is (1 2 1)/4 x (1 2 1)/4: across z and y (v_x) or z and x (v_y) the in-plane part
// is summed from shared memory and the z part from the thread's last planes; v_z takes nine
// values of its plane.  Products with the Roe weight sqrt(rho) of plane k - 1 then meet their
// neighbours through shared memory, remapped so that each face row is stored contiguously.
// One plane of loads is in flight ahead.  Bound by its two barriers a plane (286 instructions
// a cell, issue 66 % busy); 166 us at 256^3.
template <bool SPECIAL>  // mirrored or prescribed ghosts may occur
__device__ __forceinline__ void face_velocity_tile(const MarchArgs<float>& A, const TileGeom& tg,
                                                   const TileMaps32& M, const float th[3],
                                                   float (*vel)[3][FV_PLANE], float (*prod)[FV_PLANE],
                                                   float* __restrict__ face) {
  const int t = threadIdx.x;
  const bool col = t < FV_PLANE;
  const int i = col ? t % FV_W - 1 : 0, j = col ? t / FV_W - 1 : 0;
  const bool in_i = i >= 0 && i < TB, in_j = j >= 0 && j < TB;
  const bool one_point = (A.flags & PPML_VHAT_1PT) != 0;
  const int base = M.off[0][i + TH] + M.off[1][j + TH];
  const bool fx = SPECIAL && M.flip[0][i + TH], fy = SPECIAL && M.flip[1][j + TH];
  int inf_xy = -1;
  if (SPECIAL) {
    inf_xy = M.inflow[1][j + TH];
    if (inf_xy < 0) inf_xy = M.inflow[0][i + TH];
  }
  auto load = [&](int k, float q[4]) {
    const int o = base + M.off[2][k + TH];
#pragma unroll
    for (int f = 0; f < 4; f++) q[f] = __ldg(A.u[f] + o);
    if (SPECIAL) {
      if (fx) q[1] = -q[1];
      if (fy) q[2] = -q[2];
      if (M.flip[2][k + TH]) q[3] = -q[3];
      int face_in = M.inflow[2][k + TH];  // the later axis decides
      if (face_in < 0) face_in = inf_xy;
      if (face_in >= 0)
#pragma unroll
        for (int f = 0; f < 4; f++) q[f] = __ldg(A.inflow + 6 * face_in + f);
    }
  };
  float next[4] = {1.0f, 0.0f, 0.0f, 0.0f};
  if (col) load(-1, next);
  float ax0 = 0.0f, ax1 = 0.0f, by0 = 0.0f, by1 = 0.0f;  // in-plane sums of planes k-2, k-1
  float vx1 = 0.0f, vy1 = 0.0f, sq1 = 1.0f, pz1 = 0.0f;  // of plane k-1
  const int me = t;
#pragma unroll 2
  for (int k = -1; k <= TB; k++) {
    const float ir = rcp_approx(next[0]), sq = sqrt_approx(next[0]);
    const float vx = next[1] * ir, vy = next[2] * ir, vz = next[3] * ir;
    float* const px = vel[k & 1][0];
    float* const py = vel[k & 1][1];
    float* const pz = vel[k & 1][2];
    if (col) {
      px[me] = vx;
      py[me] = vy;
      pz[me] = vz;
      if (k < TB) load(k + 1, next);
    }
    __syncthreads();
    // (k = -1: only the sums of the plane)
    float ax = 4.0f * vx, by = 4.0f * vy, vt = vz;
    if (col && !one_point) {
      if (in_j) ax = 2.0f * vx + (px[me - FV_W] + px[me + FV_W]);
      if (in_i) by = 2.0f * vy + (py[me - 1] + py[me + 1]);
      if (in_i && in_j)
        vt = 0.25f * vz + 0.125f * ((pz[me - 1] + pz[me + 1]) + (pz[me - FV_W] + pz[me + FV_W])) +
             0.0625f * ((pz[me - FV_W - 1] + pz[me - FV_W + 1]) +
                        (pz[me + FV_W - 1] + pz[me + FV_W + 1]));
    }
    const float pzk = vt * sq;
    if (k >= 0 && in_i && in_j && col)  // face between k-1 and k
      face[2 * FACE_AXIS + k * TN + i + TB * j] = th[2] * ((pzk + pz1) * rcp_approx(sq + sq1));
    if (k >= 1) {  // plane k - 1 is complete
      if (col) {
        const float tx = one_point ? vx1 : 0.0625f * (2.0f * ax1 + (ax0 + ax));
        const float ty = one_point ? vy1 : 0.0625f * (2.0f * by1 + (by0 + by));
        prod[0][me] = tx * sq1;
        prod[1][me] = ty * sq1;
        prod[2][me] = sq1;
      }
      __syncthreads();
      if (t < (TB + 1) * TB) {
        const int l = t % TB, f = t / TB;  // line, face
        const int ex = (l + 1) * FV_W + f;  // x face f of row y = l: cells f-1 and f
        const float wx = (prod[0][ex] + prod[0][ex + 1]) * rcp_approx(prod[2][ex] + prod[2][ex + 1]);
        face[f * TN + l + TB * (k - 1)] = th[0] * wx;
        const int ey = f * FV_W + l + 1;  // y face f of column x = l
        const float wy =
            (prod[1][ey] + prod[1][ey + FV_W]) * rcp_approx(prod[2][ey] + prod[2][ey + FV_W]);
        face[FACE_AXIS + f * TN + l + TB * (k - 1)] = th[1] * wy;
      }
    }
    ax0 = ax1;
    ax1 = ax;
    by0 = by1;
    by1 = by;
    vx1 = vx;
    vy1 = vy;
    sq1 = sq;
    pz1 = pzk;
  }
}

__global__ void __launch_bounds__(FV_THREADS, 4) face_velocity_f32(MarchArgs<float> A) {
  __shared__ float vel[2][3][FV_PLANE];
  __shared__ float prod[3][FV_PLANE];
  __shared__ TileMaps32 maps;
  const int tiles[3] = {A.tiles_x, A.tiles_y, A.tiles_z};
  const TileGeom tg = tile_geom(A.g, tiles, A.tile_order, A.tile_first + blockIdx.x);
  if (!tg.valid) return;
  build_maps32(maps, A.g, tg);
  double stc[4];
  cta_step_constants(A.dt_dev, A.dt_host, A.h, stc);  // (a barrier: the maps are built)
  const float th[3] = {(float)stc[1], (float)stc[2], (float)stc[3]};
  float* const face = A.face + (size_t)(tg.id - A.face_first) * FACE_TILE;
  if (!tg.fast && (A.any_reflect || A.any_inflow))
    face_velocity_tile<true>(A, tg, maps, th, vel, prod, face);
  else
    face_velocity_tile<false>(A, tg, maps, th, vel, prod, face);
}

// ----------------------------------------------------------------------------- the sweeps

// One line of two fields: q(p) for the positions -3..18 (called in order, each once), w(c) the
// face velocities 0..16 (in order); emit(c, d, qc) for the cells c = 0..15 with
// d = th (F+ - F-).  ahead() is called before the last four steps: the place to issue the
// loads that the next sweep starts with.
template <bool FLAT, typename QF, typename WF, typename EF, typename AF>
__device__ __forceinline__ void lag_line_pair(QF q, WF w, EF emit, AF ahead) {
  LinePair<FLAT> ln;
  {
    const float2 a = q(-3), b = q(-2), c = q(-1);
    ln.start(a, b, c);
  }
  ln.push(q(0));
  ln.push(q(1));
  float2 ql = ln.q2, Ll = ln.Pl, Lr = ln.Pr;
  ln.push(q(2));
  float2 Fp = upwind_flux_pair(w(0), ql, Ll, Lr, ln.q2, ln.Pl, ln.Pr);
  ql = ln.q2;
  Ll = ln.Pl;
  Lr = ln.Pr;
  auto step = [&](int c) {
    ln.push(q(c + 3));
    const float2 F = upwind_flux_pair(w(c + 1), ql, Ll, Lr, ln.q2, ln.Pl, ln.Pr);
    emit(c, sub2(F, Fp), ql);
    Fp = F;
    ql = ln.q2;
    Ll = ln.Pl;
    Lr = ln.Pr;
  };
#pragma unroll
  for (int c0 = 0; c0 < TB - 4; c0 += 4) {
#pragma unroll
    for (int k = 0; k < 4; k++) step(c0 + k);
  }
  ahead();
#pragma unroll
  for (int c = TB - 4; c < TB; c++) step(c);
}

struct SweepSmem {
  float2 core[ACC];  // two fields, pitches 17 and 272: every sweep's 8-byte accesses of a
  float2 acc[ACC];   // half warp fall on 16 different bank pairs
};

// The sweeps of a tile, two fields at a time.  The z sweep reads the thread's column from
// global memory eight positions ahead and leaves the core and its divergence in shared
// memory; the x sweep adds its divergence there; the y sweep finishes into the output, rows
// of x.  The x and y lines of a warp lie in the warp's own two
// z planes, so between them only the warp meets.  Each sweep issues the first loads of the
// next (halos, face velocities) before its last four steps.
// SPECIAL: mirrored or prescribed ghosts may occur.
template <bool FLAT, bool SPECIAL>
__device__ __forceinline__ void sweep_tile(const MarchArgs<float>& A, const TileGeom& tg,
                                           const TileMaps32& maps, SweepSmem& S,
                                           const float* __restrict__ face, int out0, int nvalid) {
  const GridGeom& g = A.g;
  const int a = threadIdx.x % TB, b = threadIdx.x / TB, nx = g.n[0];
  // the thread's lines: z (x = a, y = b), x (y = a, z = b), y (x = a, z = b)
  const int zbase = maps.off[0][a + TH] + maps.off[1][b + TH];
  const int xbase = maps.off[1][a + TH] + maps.off[2][b + TH];
  const int ybase = maps.off[0][a + TH] + maps.off[2][b + TH];
  // cells of the core beyond the domain's x and y ends are ghosts to the x and y sweeps:
  // columns there carry the mirrors and prescribed states of those axes
  const bool col_fx = SPECIAL && maps.flip[0][a + TH], col_fy = SPECIAL && maps.flip[1][b + TH];
  int col_in = -1;
  if (SPECIAL) {
    col_in = maps.inflow[1][b + TH];
    if (col_in < 0) col_in = maps.inflow[0][a + TH];
  }
  // fields f, f + 1 at position p of the line with offset base along ax, through the maps
  auto fetch = [&](int f, int ax, int base, int p) {
    const int o = base + maps.off[ax][p + TH];
    float2 v = make_float2(__ldg(A.u[f] + o), __ldg(A.u[f + 1] + o));
    if (SPECIAL) {
      if (maps.flip[ax][p + TH]) {
        if (f == 1 + ax) v.x = -v.x;
        if (f == ax) v.y = -v.y;
      }
      int in = maps.inflow[ax][p + TH];
      if (ax == 2) {
        if (col_fx && f == 0) v.y = -v.y;  // m_x
        if (col_fy && f == 2) v.x = -v.x;  // m_y
        if (in < 0) in = col_in;           // (the later axis decides)
      }
      if (in >= 0) v = make_float2(__ldg(A.inflow + 6 * in + f), __ldg(A.inflow + 6 * in + f + 1));
    }
    return v;
  };
  const float* const wx = face;
  const float* const wy = face + FACE_AXIS;
  const float* const wz = face + 2 * FACE_AXIS;
  float2 ring[8], halo[6], yhalo[6];
  float wr[4], wn[4];  // face velocities: ring of the running sweep, first four of the next
  auto first_w = [&](const float* w) {
#pragma unroll
    for (int c = 0; c < 4; c++) wn[c] = __ldg(w + c * TN);
  };
  auto take_w = [&]() {
#pragma unroll
    for (int c = 0; c < 4; c++) wr[c] = wn[c];
  };
  auto ring_w = [&](const float* w, int c) {
    const float v = wr[c & 3];
    if (c + 4 <= TB) wr[c & 3] = __ldg(w + (c + 4) * TN);
    return v;
  };
  auto first_z = [&](int f) {
#pragma unroll
    for (int p = 0; p < 8; p++) ring[p] = fetch(f, 2, zbase, p - TH);
    first_w(wz);
  };
  auto low_halo = [&](int f, int ax, int base) {  // positions -3..-1
#pragma unroll
    for (int h = 0; h < 3; h++) halo[h] = fetch(f, ax, base, h - 3);
    first_w(ax == 0 ? wx : wy);
  };
  auto high_halo = [&](int f, int ax, int base) {  // positions 16..18
#pragma unroll
    for (int h = 3; h < 6; h++) halo[h] = fetch(f, ax, base, TB + h - 3);
  };
  auto line_q = [&](const float2* core, int stride, int p) {  // x and y lines
    if (p < 0) return halo[p < -2 ? 0 : (p < -1 ? 1 : 2)];
    if (p < TB) return core[p * stride];
    return p == TB ? halo[3] : (p == TB + 1 ? halo[4] : halo[5]);
  };
  first_z(0);
#pragma unroll 1
  for (int f = 0; f < 6; f += 2) {
    {  // z
      float2* const core = &S.core[acc_at(a, b, 0)];
      float2* const acc = &S.acc[acc_at(a, b, 0)];
      take_w();
      lag_line_pair<FLAT>(
          [&](int p) {
            const float2 v = ring[(p + 3) & 7];
            if (p + 8 < TB + TH) ring[(p + 3) & 7] = fetch(f, 2, zbase, p + 8);
            if (p >= 0 && p < TB) core[p * APP] = v;
            return v;
          },
          [&](int c) { return ring_w(wz, c); },
          [&](int c, float2 d, float2) { acc[c * APP] = d; },
          [&]() {
            low_halo(f, 0, xbase);
            high_halo(f, 0, xbase);
          });
    }
#pragma unroll
    for (int h = 0; h < 6; h++) yhalo[h] = fetch(f, 1, ybase, h < 3 ? h - 3 : TB + h - 3);
    __syncthreads();
    {  // x
      const float2* const core = &S.core[acc_at(0, a, b)];
      float2* const acc = &S.acc[acc_at(0, a, b)];
      take_w();
      lag_line_pair<FLAT>([&](int p) { return line_q(core, 1, p); },
                          [&](int c) { return ring_w(wx, c); },
                          [&](int c, float2 d, float2) { acc[c] = add2(acc[c], d); },
                          [&]() { first_w(wy); });
    }
#pragma unroll
    for (int h = 0; h < 6; h++) halo[h] = yhalo[h];
    __syncwarp();
    {  // y
      const float2* const core = &S.core[acc_at(a, 0, b)];
      const float2* const acc = &S.acc[acc_at(a, 0, b)];
      float* const o0 = A.out[f] + out0;
      float* const o1 = A.out[f + 1] + out0;
      take_w();
      lag_line_pair<FLAT>([&](int p) { return line_q(core, ARP, p); },
                          [&](int c) { return ring_w(wy, c); },
                          [&](int c, float2 d, float2 qc) {
                            if (c < nvalid) {
                              const float2 v = sub2(qc, add2(acc[c * ARP], d));
                              o0[(size_t)c * nx] = v.x;
                              o1[(size_t)c * nx] = v.y;
                            }
                          },
                          [&]() {
                            if (f < 4) first_z(f + 2);
                          });
    }
    __syncthreads();  // the next z sweep writes the core and the accumulator
  }
}

template <bool FLAT>
__global__ void __launch_bounds__(TN, 2) lagrangian_sweep_f32(MarchArgs<float> A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SweepSmem& S = *reinterpret_cast<SweepSmem*>(smem_raw);
  __shared__ TileMaps32 maps;
  const GridGeom& g = A.g;
  const int tid = threadIdx.x, a = tid % TB, b = tid / TB;
  const int tiles[3] = {A.tiles_x, A.tiles_y, A.tiles_z};
  const TileGeom tg = tile_geom(g, tiles, A.tile_order, A.tile_first + blockIdx.x);
  if (!tg.valid) return;  // a padding block of a blocked order (uniform over the CTA)
  build_maps32(maps, g, tg);
  __syncthreads();
  const float* const face = A.face + (size_t)(tg.id - A.face_first) * FACE_TILE + tid;
  const bool line_ok = tg.i0 + a < g.n[0] && tg.k0 + b < g.n[2];
  const int nvalid = line_ok ? min(TB, g.n[1] - tg.j0) : 0;
  const int nx = g.n[0];
  const int out0 = (tg.i0 + a) + nx * tg.j0 + (int)g.nxy * (tg.k0 + b);
  if (!tg.fast && (A.any_reflect || A.any_inflow))
    sweep_tile<FLAT, true>(A, tg, maps, S, face, out0, nvalid);
  else
    sweep_tile<FLAT, false>(A, tg, maps, S, face, out0, nvalid);

  // ---- energy correction (Sec. 1.4), CFL maxima and sums of the thread's y line
  FieldSums<float> sums;
  sums.init();
  float vmax = 0.0f, cmax = 0.0f;
  unsigned long long nvac = 0, nbad = 0;
  const float gamma = (float)A.gamma, gm1 = (float)(A.gamma - 1.0);
  const float rho_vac_up = __double2float_ru(A.rho_vac);
  constexpr int FB = 2;  // cells at a time, the next ones' loads in flight
  float nu[FB][6];
  auto load = [&](int c0) {
#pragma unroll
    for (int q = 0; q < FB; q++) {
      const size_t idx = out0 + (size_t)min(c0 + q, nvalid - 1) * nx;
#pragma unroll
      for (int f = 0; f < 6; f++) nu[q][f] = A.out[f][idx];
    }
  };
  if (nvalid > 0) load(0);
#pragma unroll 1
  for (int c0 = 0; c0 < nvalid; c0 += FB) {
    float u[FB][6];
#pragma unroll
    for (int q = 0; q < FB; q++)
#pragma unroll
      for (int f = 0; f < 6; f++) u[q][f] = nu[q][f];
    if (c0 + FB < nvalid) load(c0 + FB);
    bool vac[FB], any_vac = false;
#pragma unroll
    for (int q = 0; q < FB; q++) {
      vac[q] = c0 + q < nvalid && vacuum_cell_f32(u[q], rho_vac_up);
      any_vac |= vac[q];
      const float e = dense_eps_f32(u[q]);
      u[q][5] = vac[q] ? u[q][5] : e;
    }
    if (any_vac) {
#pragma unroll
      for (int q = 0; q < FB; q++)
        if (vac[q]) {
          vacuum_correct_f32(u[q], A.rho_vac);
          nvac++;
        }
    }
#pragma unroll
    for (int q = 0; q < FB; q++) {
      if (c0 + q >= nvalid) break;
      const size_t idx = out0 + (size_t)(c0 + q) * nx;
      if (vac[q]) {
#pragma unroll
        for (int f = 1; f <= 3; f++) A.out[f][idx] = u[q][f];
      }
      A.out[5][idx] = u[q][5];
      sums.add(u[q]);
      cell_speeds_f32(u[q], gamma, gm1, vmax, cmax, nbad);
    }
  }
  float hi[6], lo[6];
#pragma unroll
  for (int f = 0; f < 6; f++) {
    hi[f] = sums.s[f].hi;
    lo[f] = sums.s[f].lo;
  }
  block_reduce_store_f32<TN>(hi, lo, vmax, cmax, (unsigned)nvac, (unsigned)nbad, A.partials, tg.id);
  finalize_last(A.partials, tiles[0] * tiles[1] * tiles[2], A.fin, read_tau(A.dt_dev, A.dt_host));
}

// ------------------------------------------------------------------------- Eulerian stage

struct EulerSmem {
  float2 re[ACC];   // (rho, rho eps) of the tile
  float mx[ACC];    // m_x of the tile, then its update
  float2 acc[ACC];  // sums over axes of th (PV+ - PV-) and th (V+ - V-)
};

// One line of the Eulerian stage, (v, p) as a packed pair of lines: q(p, v, r) gives the pair
// (v_a, p) and rho at the positions p = -3..18 (called in order, each once).  emit(c, dm, dpv,
// dv) for the cells c = 0 .. 15 as sweep_eulerian_faces describes.  ahead(): before the last four steps.
template <bool FLAT, typename QF, typename EF, typename AF>
__device__ __forceinline__ void euler_line_pair(QF q, float gamma, float th, EF emit, AF ahead) {
  LinePair<FLAT> ln;
  float r1, r2, rn, skip;  // rho at p-1, p-2, p
  {
    float2 a, b, c;
    q(-3, a, skip);
    q(-2, b, skip);
    q(-1, c, r2);
    ln.start(a, b, c);
  }
  {
    float2 v;
    q(0, v, r1);
    ln.push(v);
    q(1, v, rn);
    ln.push(v);
  }
  FaceCell left{ln.q2, ln.Pl, ln.Pr};  // cell p-3, the face's left cell
  face_roots(left, r2);
  r2 = r1;
  r1 = rn;
  float Vp = 0.0f, Pp = 0.0f;
  auto face = [&](int p, float& V, float& P) {  // after position p: the face of p-3 and p-2
    float2 v;
    q(p, v, rn);
    ln.push(v);
    FaceCell right{ln.q2, ln.Pl, ln.Pr};
    face_roots(right, r2);
    acoustic_face(left, right, gamma, th, V, P);
    left = right;
    r2 = r1;
    r1 = rn;
  };
  face(2, Vp, Pp);
  auto step = [&](int c) {
    float V, P;
    face(c + 3, V, P);
    emit(c, th * (P - Pp), th * (P * V - Pp * Vp), th * (V - Vp));
    Vp = V;
    Pp = P;
  };
#pragma unroll 1
  for (int c0 = 0; c0 < TB - 4; c0 += 4) {
#pragma unroll
    for (int k = 0; k < 4; k++) step(c0 + k);
  }
  ahead();
#pragma unroll
  for (int c = TB - 4; c < TB; c++) step(c);
}

// The Eulerian stage of a tile.  The z sweep reads rho, rho eps and m_z of the thread's column
// from global memory, stores m_z's update and leaves (rho, rho eps), m_x and its pressure-work
// and divergence terms in shared memory; the x sweep reads the core there and leaves m_x's
// update in place; the y sweep reads m_y in rows of x, adds its terms and stores m_x, m_y,
// rho E and rho eps, all in rows of x.  One CTA barrier: the x and y lines of a warp lie in
// its own two z planes.  PHI: the gravity source terms, each where its momentum is at hand.
// SPECIAL: mirrored or prescribed ghosts may occur.
template <bool FLAT, bool PHI, bool SPECIAL>
__device__ __forceinline__ void euler_tile(const MarchArgs<float>& A, const TileGeom& tg,
                                           const TileMaps32& maps, EulerSmem& S,
                                           const float th[3], float tau) {
  const GridGeom& g = A.g;
  const int a = threadIdx.x % TB, b = threadIdx.x / TB, nx = g.n[0], nxy = (int)g.nxy;
  const float gamma = (float)A.gamma, gm1 = (float)(A.gamma - 1.0);
  const int zbase = maps.off[0][a + TH] + maps.off[1][b + TH];
  const int xbase = maps.off[1][a + TH] + maps.off[2][b + TH];
  const int ybase = maps.off[0][a + TH] + maps.off[2][b + TH];
  // ghost cells of the core beyond the domain's x and y ends (see sweep_tile)
  const bool col_fx = SPECIAL && maps.flip[0][a + TH];
  int col_in = -1;
  if (SPECIAL) {
    col_in = maps.inflow[1][b + TH];
    if (col_in < 0) col_in = maps.inflow[0][a + TH];
  }
  // rho, m_ax and rho eps at position p of the line with offset base along ax
  auto fetch = [&](int ax, int base, int p) {
    const int o = base + maps.off[ax][p + TH];
    float3 v = make_float3(__ldg(A.u[0] + o), __ldg(A.u[1 + ax] + o), __ldg(A.u[5] + o));
    if (SPECIAL) {
      if (maps.flip[ax][p + TH]) v.y = -v.y;
      int in = maps.inflow[ax][p + TH];
      if (ax == 2 && in < 0) in = col_in;
      if (in >= 0)
        v = make_float3(__ldg(A.inflow + 6 * in), __ldg(A.inflow + 6 * in + 1 + ax),
                        __ldg(A.inflow + 6 * in + 5));
    }
    return v;
  };
  auto fetch_mx = [&](int p) {  // m_x of the column's cell p of the core
    float m = __ldg(A.u[1] + (zbase + maps.off[2][p + TH]));
    if (SPECIAL) {
      if (col_fx) m = -m;
      int in = maps.inflow[2][p + TH];
      if (in < 0) in = col_in;
      if (in >= 0) m = __ldg(A.inflow + 6 * in + 1);
    }
    return m;
  };
  // Phi's neighbour along ax at coordinate c (domain) in direction dir, as an offset: wraps at
  // periodic faces, zero-gradient at the others
  auto phi_step = [&](int ax, int c, int dir) {
    const int n = g.n[ax], q = c + dir, st = ax == 0 ? 1 : (ax == 1 ? nx : nxy);
    if ((unsigned)q < (unsigned)n) return dir * st;
    return g.bc[2 * ax + (dir > 0)] == PPML_BC_PERIODIC ? -dir * (n - 1) * st : 0;
  };
  float3 ring[4], halo[6], yhalo[6];
  float mring[4];
  // ---- z
  {
    float2* const re = &S.re[acc_at(a, b, 0)];
    float* const mx = &S.mx[acc_at(a, b, 0)];
    float2* const acc = &S.acc[acc_at(a, b, 0)];
    const bool ok = tg.i0 + a < nx && tg.j0 + b < g.n[1];
    const int nvalid = ok ? min(TB, g.n[2] - tg.k0) : 0;
    const int o0 = (tg.i0 + a) + nx * (tg.j0 + b) + nxy * tg.k0;
    float* const om = A.out[3] + o0;
    const float rg = PHI ? tau / (float)(2.0 * A.h[2]) : 0.0f;
    float m1 = 0.0f, m2 = 0.0f, m3 = 0.0f, mn = 0.0f;  // m_z at p-1, p-2, p-3, p
    float d1 = 0.0f, d2 = 0.0f, d3 = 0.0f, dn = 0.0f;  // rho there (PHI)
#pragma unroll
    for (int p = 0; p < 4; p++) ring[p] = fetch(2, zbase, p - TH);
#pragma unroll
    for (int p = 0; p < 4; p++) mring[p] = fetch_mx(p);
    euler_line_pair<FLAT>(
        [&](int p, float2& v, float& r) {
          const float3 u = ring[(p + 3) & 3];
          if (p + 4 < TB + TH) ring[(p + 3) & 3] = fetch(2, zbase, p + 4);
          if (p >= 0 && p < TB) {
            re[p * APP] = make_float2(u.x, u.z);
            mx[p * APP] = mring[p & 3];
            if (p + 4 < TB) mring[p & 3] = fetch_mx(p + 4);
          }
          v = make_float2(u.y * rcp_approx(u.x), gm1 * u.z);
          r = u.x;
          m3 = m2;
          m2 = m1;
          m1 = mn;
          mn = u.y;
          if (PHI) {
            d3 = d2;
            d2 = d1;
            d1 = dn;
            dn = u.x;
          }
        },
        gamma, th[2],
        [&](int c, float dm, float dpv, float dv) {
          if (PHI && c < nvalid) {
            const float* const f = A.phi + o0 + (size_t)c * nxy;
            const float gr = (__ldg(f + phi_step(2, tg.k0 + c, 1)) - __ldg(f + phi_step(2, tg.k0 + c, -1))) * rg;
            dm = fmaf(d3, gr, dm);
            dpv = fmaf(m3, gr, dpv);
          }
          acc[c * APP] = make_float2(dpv, dv);
          if (c < nvalid) om[(size_t)c * nxy] = m3 - dm;
        },
        [&]() {
#pragma unroll
          for (int h = 0; h < 6; h++) halo[h] = fetch(0, xbase, h < 3 ? h - 3 : TB + h - 3);
        });
  }
#pragma unroll
  for (int h = 0; h < 6; h++) yhalo[h] = fetch(1, ybase, h < 3 ? h - 3 : TB + h - 3);
  __syncthreads();
  const bool yok = tg.i0 + a < nx && tg.k0 + b < g.n[2];
  const int nvalid = yok ? min(TB, g.n[1] - tg.j0) : 0;
  const int o0 = (tg.i0 + a) + nx * tg.j0 + nxy * (tg.k0 + b);  // the y line's first cell
  auto my_at = [&](int p) { return __ldg(A.u[2] + (ybase + maps.off[1][p + TH])); };
  float ering[4];
  // ---- x
  {
    const float2* const re = &S.re[acc_at(0, a, b)];
    float* const mx = &S.mx[acc_at(0, a, b)];
    float2* const acc = &S.acc[acc_at(0, a, b)];
    euler_line_pair<FLAT>(
        [&](int p, float2& v, float& r) {
          float3 u;
          if (p < 0 || p >= TB) {
            u = p < 0 ? halo[p < -2 ? 0 : (p < -1 ? 1 : 2)]
                      : (p == TB ? halo[3] : (p == TB + 1 ? halo[4] : halo[5]));
          } else {
            const float2 q = re[p];
            u = make_float3(q.x, mx[p], q.y);
          }
          v = make_float2(u.y * rcp_approx(u.x), gm1 * u.z);
          r = u.x;
        },
        gamma, th[0],
        [&](int c, float dm, float dpv, float dv) {
          acc[c] = add2(acc[c], make_float2(dpv, dv));
          mx[c] = mx[c] - dm;
        },
        [&]() {
#pragma unroll
          for (int p = 0; p < 4; p++) {
            mring[p] = my_at(p);
            ering[p] = p < nvalid ? __ldg(A.u[4] + o0 + (size_t)p * nx) : 0.0f;
          }
        });
  }
#pragma unroll
  for (int h = 0; h < 6; h++) halo[h] = yhalo[h];
  __syncwarp();
  // ---- y
  {
    const float2* const re = &S.re[acc_at(a, 0, b)];
    const float* const mx = &S.mx[acc_at(a, 0, b)];
    const float2* const acc = &S.acc[acc_at(a, 0, b)];
    const float rgx = PHI ? tau / (float)(2.0 * A.h[0]) : 0.0f;
    const float rgy = PHI ? tau / (float)(2.0 * A.h[1]) : 0.0f;
    const int pxm = PHI ? phi_step(0, tg.i0 + a, -1) : 0, pxp = PHI ? phi_step(0, tg.i0 + a, 1) : 0;
    float m1 = 0.0f, m2 = 0.0f, m3 = 0.0f, mn = 0.0f;  // m_y at p-1, p-2, p-3, p
    euler_line_pair<FLAT>(
        [&](int p, float2& v, float& r) {
          float3 u;
          if (p < 0 || p >= TB) {
            u = p < 0 ? halo[p < -2 ? 0 : (p < -1 ? 1 : 2)]
                      : (p == TB ? halo[3] : (p == TB + 1 ? halo[4] : halo[5]));
          } else {
            const float2 q = re[p * ARP];
            float m = mring[p & 3];
            if (SPECIAL) {  // core cells beyond the domain's y end are ghosts of this sweep
              if (maps.flip[1][p + TH]) m = -m;
              const int in = maps.inflow[1][p + TH];
              if (in >= 0) m = __ldg(A.inflow + 6 * in + 2);
            }
            if (p + 4 < TB) mring[p & 3] = my_at(p + 4);
            u = make_float3(q.x, m, q.y);
          }
          v = make_float2(u.y * rcp_approx(u.x), gm1 * u.z);
          r = u.x;
          m3 = m2;
          m2 = m1;
          m1 = mn;
          mn = u.y;
        },
        gamma, th[1],
        [&](int c, float dm, float dpv, float dv) {
          const float en = ering[c & 3];
          if (c + 4 < nvalid) ering[c & 3] = __ldg(A.u[4] + o0 + (size_t)(c + 4) * nx);
          if (c < nvalid) {
            const float2 s = acc[c * ARP], q = re[c * ARP];
            const size_t o = o0 + (size_t)c * nx;
            float m = mx[c * ARP];
            if (PHI) {
              const float* const f = A.phi + o;
              const int j = tg.j0 + c;
              const float gy = (__ldg(f + phi_step(1, j, 1)) - __ldg(f + phi_step(1, j, -1))) * rgy;
              const float gx = (__ldg(f + pxp) - __ldg(f + pxm)) * rgx;
              dm = fmaf(q.x, gy, dm);
              dpv = fmaf(m3, gy, dpv);
              m = fmaf(-q.x, gx, m);
              dpv = fmaf(__ldg(A.u[1] + o), gx, dpv);
            }
            A.out[1][o] = m;
            A.out[2][o] = m3 - dm;
            A.out[4][o] = en - (s.x + dpv);
            A.out[5][o] = eps_update(q.y, gm1, s.y + dv);
            if (A.out[0]) A.out[0][o] = q.x;
          }
        },
        [&]() {});
  }
}

template <bool FLAT, bool PHI>
__global__ void __launch_bounds__(TN, 2) eulerian_sweep_f32(MarchArgs<float> A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  EulerSmem& S = *reinterpret_cast<EulerSmem*>(smem_raw);
  __shared__ TileMaps32 maps;
  const int tiles[3] = {A.tiles_x, A.tiles_y, A.tiles_z};
  const TileGeom tg = tile_geom(A.g, tiles, A.tile_order, blockIdx.x);
  if (!tg.valid) return;  // a padding block of a blocked order (uniform over the CTA)
  build_maps32(maps, A.g, tg);
  double stc[4];
  cta_step_constants(A.dt_dev, A.dt_host, A.h, stc);  // (a barrier: the maps are built)
  const float th[3] = {(float)stc[1], (float)stc[2], (float)stc[3]};
  if (!tg.fast && (A.any_reflect || A.any_inflow))
    euler_tile<FLAT, PHI, true>(A, tg, maps, S, th, (float)stc[0]);
  else
    euler_tile<FLAT, PHI, false>(A, tg, maps, S, th, (float)stc[0]);
}

}  // namespace ppml
