// Isolated-boundary Poisson solve of the paper's Sec. "The Poisson solver" (Stages 1-3 with
// the 27-point stencil, eq. stencil27point).
//
// Stage 1: the monopole and quadrupole moments of the cell masses about the coordinate
// centre (a deterministic FP64 reduction) give the potential on the shell of cells just
// outside the grid (MacCullagh's formula, with its factor 1/2); the shell values that enter
// the stencil of a boundary cell are moved to the right-hand side.  Stages 2-3: with
// Dirichlet data on the shell the 27-point operator is diagonal in the sine basis
// sin(pi j (i + 1) / (N + 1)), j = 1..N, so the exponential transform the paper prints is
// replaced by a type-I sine transform along each axis (FP32 grids of at most 256 points per
// axis: dense half-size matrix products; else odd extension to 2 (N + 1) points and a batched
// real-to-complex cuFFT), the amplitudes are divided by the operator's eigenvalue
// 6 (prod_a (1 - (2/3) sin^2(pi j_a / (2 (N_a + 1)))) - 1), and the same sine transform,
// scaled by prod_a 2 / (N_a + 1), brings the potential back.  The right-hand side is
// 4 pi G h^2 (rho + D7 rho / 12) (D7 the 7-point second difference, rho = 0 outside), which
// makes the 27-point solve fourth-order accurate as the paper states; the printed
// 4 pi G h^2 rho (second order) is available with PPML_POISSON_PRINTED_RHS.
//
// Geometry: cell (i, j, k) has its centre at ((i + 1/2 - nx/2) h, (j + 1/2 - ny/2) h,
// (k + 1/2 - nz/2) h), i.e. the grid is centred on the origin of the expansion.
//
// The potential array doubles as the work array of the transforms; the sine matrices, or the
// odd extension and the half spectrum, live in buffers kept by the solver state between calls.
//
// FP32 grids form the moments, the source and the symbol in float pairs (about 2^-45, below
// the float potential's rounding), off the FP64 pipe, where the values lie in the pairs'
// range, else in double.
#include <cuda_runtime.h>
#include <cufft.h>
#include <float.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "../../include/ppml.h"
#include "ppml_pair.cuh"
#include "ppml_internal.h"

using namespace ppml;

namespace {

constexpr int kThreads = 256;
constexpr int kMoments = 7;  // M, I_x, I_y, I_z, I_xy, I_xz, I_yz
constexpr int kMaxMomentBlocks = 1216;  // 8 per SM on 152 SMs

struct Dims {
  int n[3];
  long long nxy, ncell;
};

__device__ __forceinline__ double centre(int i, int n, double h) {
  return ((double)i + 0.5 - 0.5 * (double)n) * h;
}

// How rows of x are spread over threads: a group of `lanes` threads (a power of two: short
// rows share a warp) takes a piece of at most `length` cells of one row, `pieces` to a row
// (more than one where the rows are fewer than the groups that should be busy, of at least
// `cells` cells a thread).
struct RowPieces {
  int log_lanes, pieces, length;
  IndexDivisor by_pieces, by_ny;
  unsigned items;  // pieces of all rows
};
RowPieces row_pieces(int nx, int ny, long long rows, long long threads, int cells) {
  int log_lanes = 0;
  while ((1 << log_lanes) < nx && log_lanes < 5) log_lanes++;
  const long long lanes = 1 << log_lanes;
  const long long most = (nx + cells * lanes - 1) / (cells * lanes);
  const int pieces = (int)std::min(std::max(1LL, threads / lanes / rows), most);
  const int length = (int)(((nx + pieces - 1) / pieces + lanes - 1) / lanes * lanes);
  return {log_lanes, pieces, length, IndexDivisor(pieces), IndexDivisor(ny), (unsigned)(rows * pieces)};
}
// The rows of a kernel's threads: WARP, rows of a warp each (a constant step).
template <bool WARP>
struct RowWalk {
  int step, lane;
  unsigned first, groups;
  __device__ __forceinline__ explicit RowWalk(const RowPieces& R) {
    const int log_lanes = WARP ? 5 : R.log_lanes;
    const unsigned per_block = kThreads >> log_lanes;
    step = 1 << log_lanes;
    lane = threadIdx.x & (step - 1);
    first = blockIdx.x * per_block + (threadIdx.x >> log_lanes);
    groups = gridDim.x * per_block;
  }
};
// The copies of the sine transform load kBatch cells before they store any (one float a thread
// in flight is half of what the memory takes).
constexpr int kBatch = 4;
// Item q: the cells i0, i0 + step, .. < i1 of row (j, k) for this lane.
struct RowItem {
  long long row;
  int j, k, i0, i1;
};
__device__ __forceinline__ RowItem row_item(const Dims& D, const RowPieces& R, unsigned q, int lane) {
  const unsigned row = R.by_pieces.quotient(q), k = R.by_ny.quotient(row);
  const int i = (int)(q - row * (unsigned)R.pieces) * R.length;
  return {(long long)row, (int)(row - k * (unsigned)D.n[1]), (int)k, i + lane,
          min(i + R.length, D.n[0])};
}

// Stage 1a: per-block FP64 partial moments of the masses rho h^3, fixed block count and a
// fixed-shape tree, so the result does not depend on scheduling.  A group of threads takes a
// row (j, k), or a piece of it, at a time and sums rho, rho x, rho x^2 over it (each lane its
// own cells); y and z are the same for the whole row, so the seven moments cost seven more
// operations per lane and row instead of about 25 FP64 operations per cell (128^3 FP32: 136 us
// before, 75 so).  A warp to every row, short or not: 1024 x 1024 cells in the y-z plane took
// 2.26 ms (81 us so), 65536 x 4 x 4 1.20 ms (42).
template <typename T, bool WARP>
__global__ void __launch_bounds__(kThreads) moment_kernel(const T* __restrict__ rho, Dims D,
                                                          RowPieces R, double h,
                                                          double* __restrict__ part) {
  double acc[kMoments] = {0, 0, 0, 0, 0, 0, 0};
  const double vol = h * h * h;
  const RowWalk<WARP> W(R);
  for (unsigned q = W.first; q < R.items; q += W.groups) {
    const RowItem t = row_item(D, R, q, W.lane);
    double m0 = 0.0, m1 = 0.0, m2 = 0.0;
    for (int i = t.i0; i < t.i1; i += W.step) {
      const double x = centre(i, D.n[0], h), m = (double)rho[t.row * D.n[0] + i], mx = m * x;
      m0 += m;
      m1 += mx;
      m2 += mx * x;
    }
    const double y = centre(t.j, D.n[1], h), z = centre(t.k, D.n[2], h);
    m0 *= vol;
    m1 *= vol;
    m2 *= vol;
    acc[0] += m0;
    acc[1] += (z * z + y * y) * m0;
    acc[2] += m2 + z * z * m0;
    acc[3] += m2 + y * y * m0;
    acc[4] += y * m1;
    acc[5] += z * m1;
    acc[6] += y * z * m0;
  }
  __shared__ double s[kMoments][kThreads];
#pragma unroll
  for (int q = 0; q < kMoments; q++) s[q][threadIdx.x] = acc[q];
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
#pragma unroll
      for (int q = 0; q < kMoments; q++) s[q][threadIdx.x] += s[q][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < kMoments) part[(size_t)blockIdx.x * kMoments + threadIdx.x] = s[threadIdx.x][0];
}

// The same on FP32 grids of at most kPairMax cells along x and y, in float pairs: the centres
// are half integers times h, so x', y' and their products are exact floats there, each term is
// a product with its exact error, and the sums are TwoSum pairs (about 2^-45, far below the
// float potential).  A block takes some rows of one plane at a time; z enters once per thread
// and item, in double: about 60 FP64 instructions a warp, so grids of small planes (below
// kPairPlane) take moment_kernel unless every block has one plane only.  Planes are cut, into
// items of at least kPairItem cells, where they are fewer than kPairBlocks (two CTAs an SM): 2048 x 2048 x 1 takes 8.0 ms on one
// CTA, 44 us so, 128 planes of 128 x 256 cells 39 and 29 us.  Sums that overflow a float
// (densities of 1e26 and more) or lie where the products' errors underflow are formed again in
// double.
constexpr int kPairMax = 2048;
constexpr int kPairPlane = 512;
constexpr int kPairItem = 2048;
constexpr int kPairBlocks = 304;
struct PairSum {
  float hi, lo;
  __device__ __forceinline__ void add(float m, float c) {  // += m c
    const float p = m * c, e = fmaf(m, c, -p);
    float s, t;
    two_sum(hi, p, s, t);
    hi = s;
    lo += t + e;
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};
__global__ void __launch_bounds__(kThreads) moment_pair_kernel(const float* __restrict__ rho, Dims D,
                                                               RowPieces R, int cuts,
                                                               IndexDivisor by_cuts, double h,
                                                               double* __restrict__ part) {
  double acc[kMoments] = {0, 0, 0, 0, 0, 0, 0};
  const int step = 1 << R.log_lanes, lane = threadIdx.x & (step - 1);
  const unsigned groups = kThreads >> R.log_lanes;
  const int rows = (int)by_cuts.quotient(D.n[1] + cuts - 1);  // of an item
  const double vol = h * h * h;
  for (unsigned item = blockIdx.x; item < (unsigned)(D.n[2] * cuts); item += gridDim.x) {
    const int k = (int)by_cuts.quotient(item), j0 = (int)(item - (unsigned)(k * cuts)) * rows;
    const unsigned pieces = max(min(rows, D.n[1] - j0), 0) * R.pieces;
    PairSum s[6] = {};  // m, m x, m y, m x x, m y y, m x y
    auto cells = [&](auto add) {  // add(m, x, y) for the thread's cells of the item
      for (unsigned q = threadIdx.x >> R.log_lanes; q < pieces; q += groups) {
        const unsigned r = R.by_pieces.quotient(q);
        const int j = j0 + (int)r, i0 = (int)(q - r * (unsigned)R.pieces) * R.length;
        const float y = (float)j + 0.5f - 0.5f * (float)D.n[1];
        const float* row = rho + (long long)k * D.nxy + (long long)j * D.n[0];
        const int i1 = min(i0 + R.length, D.n[0]);
        for (int i = i0 + lane; i < i1; i += step)
          add(row[i], (float)i + 0.5f - 0.5f * (float)D.n[0], y);
      }
    };
    cells([&](float m, float x, float y) {
      s[0].add(m, 1.0f);
      s[1].add(m, x);
      s[2].add(m, y);
      s[3].add(m, x * x);
      s[4].add(m, y * y);
      s[5].add(m, x * y);
    });
    double t[6];
    bool in_range = s[0].hi == 0.0f || fabsf(s[0].hi) >= 0x1p-110f;
#pragma unroll
    for (int q = 0; q < 6; q++) {
      t[q] = s[q].value();
      in_range = in_range && fabs(t[q]) <= (double)FLT_MAX;
    }
    if (!in_range) {
#pragma unroll
      for (int q = 0; q < 6; q++) t[q] = 0.0;
      cells([&](float m, float x, float y) {
        const double dm = m, dx = dm * x, dy = dm * y;
        t[0] += dm;
        t[1] += dx;
        t[2] += dy;
        t[3] += dx * x;
        t[4] += dy * y;
        t[5] += dx * y;
      });
    }
    const double z = centre(k, D.n[2], h), m0 = vol * t[0], mx = vol * h * t[1], my = vol * h * t[2],
                 mxx = vol * h * h * t[3], myy = vol * h * h * t[4], mxy = vol * h * h * t[5];
    acc[0] += m0;
    acc[1] += z * z * m0 + myy;
    acc[2] += mxx + z * z * m0;
    acc[3] += mxx + myy;
    acc[4] += mxy;
    acc[5] += z * mx;
    acc[6] += z * my;
  }
  __shared__ double sh[kMoments][kThreads];
#pragma unroll
  for (int q = 0; q < kMoments; q++) sh[q][threadIdx.x] = acc[q];
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
#pragma unroll
      for (int q = 0; q < kMoments; q++) sh[q][threadIdx.x] += sh[q][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < kMoments) part[(size_t)blockIdx.x * kMoments + threadIdx.x] = sh[threadIdx.x][0];
}

// Stage 1b: one block folds the partials in a fixed order.
__global__ void __launch_bounds__(kThreads) moment_final_kernel(const double* __restrict__ part,
                                                                int nblk, double* __restrict__ mom) {
  __shared__ double s[kMoments][kThreads];
  double acc[kMoments] = {0, 0, 0, 0, 0, 0, 0};
  for (int b = threadIdx.x; b < nblk; b += kThreads)
#pragma unroll
    for (int q = 0; q < kMoments; q++) acc[q] += part[(size_t)b * kMoments + q];
#pragma unroll
  for (int q = 0; q < kMoments; q++) s[q][threadIdx.x] = acc[q];
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
#pragma unroll
      for (int q = 0; q < kMoments; q++) s[q][threadIdx.x] += s[q][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < kMoments) mom[threadIdx.x] = s[threadIdx.x][0];
}

// Monopole + quadrupole potential at (x, y, z) (MacCullagh's formula).
__device__ double shell_potential(const double* __restrict__ mom, double x, double y, double z,
                                  double G) {
  const double r2 = x * x + y * y + z * z;
  const double r = sqrt(r2);
  const double I0 = ((x * x * mom[1] + y * y * mom[2] + z * z * mom[3]) -
                     2.0 * (x * y * mom[4] + x * z * mom[5] + y * z * mom[6])) /
                    r2;
  return -G * mom[0] / r - 0.5 * G * (mom[1] + mom[2] + mom[3] - 3.0 * I0) / (r2 * r);
}

// Stage 1c: the potential on the shell of cells around the grid, each shell cell once (a
// boundary cell's stencil meets up to 19 of them, and consecutive threads of the right-hand
// side are mostly not boundary cells).  Layout of the (nx+2)(ny+2)(nz+2) box's surface: the
// two z planes, then per inner z the two y rows, then the two x columns.
__host__ __device__ __forceinline__ long long shell_cells(const Dims& D) {
  const long long X = D.n[0] + 2, Y = D.n[1] + 2;
  return 2 * X * Y + (long long)D.n[2] * (2 * X + 2 * D.n[1]);
}
// Index of shell cell (i, j, k), each in -1 .. n.
__device__ __forceinline__ long long shell_at(const Dims& D, int i, int j, int k) {
  const long long X = D.n[0] + 2, Y = D.n[1] + 2;
  if (k < 0 || k >= D.n[2]) return (k < 0 ? 0 : X * Y) + X * (j + 1) + (i + 1);
  const long long base = 2 * X * Y + (long long)k * (2 * X + 2 * D.n[1]);
  if (j < 0 || j >= D.n[1]) return base + (j < 0 ? 0 : X) + (i + 1);
  return base + 2 * X + (i < 0 ? 0 : D.n[1]) + j;
}
__global__ void __launch_bounds__(kThreads) shell_kernel(Dims D, double h, double G,
                                                         const double* __restrict__ mom,
                                                         double* __restrict__ shell) {
  const long long n = shell_cells(D), X = D.n[0] + 2, Y = D.n[1] + 2;
  for (long long q = (long long)blockIdx.x * kThreads + threadIdx.x; q < n;
       q += (long long)gridDim.x * kThreads) {
    int i, j, k;
    if (q < 2 * X * Y) {
      k = q < X * Y ? -1 : D.n[2];
      const int r = (int)(q % (X * Y));
      j = r / (int)X - 1;
      i = r % (int)X - 1;
    } else {
      const int per = 2 * (int)X + 2 * D.n[1];
      k = (int)((q - 2 * X * Y) / per);
      const int r = (int)((q - 2 * X * Y) % per);
      if (r < 2 * (int)X) {
        j = r < (int)X ? -1 : D.n[1];
        i = r % (int)X - 1;
      } else {
        i = r - 2 * (int)X < D.n[1] ? -1 : D.n[0];
        j = (r - 2 * (int)X) % D.n[1];
      }
    }
    shell[q] = shell_potential(mom, centre(i, D.n[0], h), centre(j, D.n[1], h),
                               centre(k, D.n[2], h), G);
  }
}

// rho + D7 rho / 12 of a cell from its value and the sum of its six neighbours.  FP32 grids
// take it as a float pair (rho / 2 + sum / 12 with the sum in TwoSum): FP64 would cost
// about 20 FP64 instructions per cell, at one per 19 cycles and SM.
struct SourcePair {
  float hi, lo;
};
__device__ __forceinline__ void pair_add(SourcePair& s, float x) {
  const float t = s.hi + x, b = t - s.hi;
  s.lo += (s.hi - (t - b)) + (x - b);
  s.hi = t;
}

// 4 pi G h^2 and, as pairs, it and its twelfth (formed once on the host: a division in each
// thread's prologue took as long as a 128^3 grid's cells).
struct Source {
  double c;
  float ch, cl, c12h, c12l;
  explicit Source(double c_) : c(c_), ch((float)c_), cl((float)(c_ - (double)ch)) {
    c12h = (float)(c / 12.0);
    c12l = (float)(c / 12.0 - (double)c12h);
  }
};

// Right-hand side 4 pi G h^2 (rho [+ D7 rho / 12]) of the cells away from the boundary, written
// into the potential array (the work array); boundary cells are left to rhs_edge_kernel.
// PAIRS: FP32 grids in float pairs, for constants in their range (ppml_pair_range); a cell
// whose pair overflows (the sum of densities above 2.8e37) is formed in double.
template <typename T, bool PAIRS, bool WARP>
__global__ void __launch_bounds__(kThreads) rhs_kernel(const T* __restrict__ rho, T* __restrict__ out,
                                                       Dims D, RowPieces R, Source S, int printed) {
  const int nx = D.n[0];
  const RowWalk<WARP> W(R);
  for (unsigned q = W.first; q < R.items; q += W.groups) {
    const RowItem t = row_item(D, R, q, W.lane);
    if (t.j == 0 || t.k == 0 || t.j == D.n[1] - 1 || t.k == D.n[2] - 1) continue;
    for (int i = t.i0; i < t.i1; i += W.step) {
      if (i == 0 || i == nx - 1) continue;
      const long long idx = t.row * nx + i;
      const T rc = rho[idx];
      T nb[6] = {};
      if (!printed) {
        nb[0] = rho[idx - 1];
        nb[1] = rho[idx + 1];
        nb[2] = rho[idx - nx];
        nb[3] = rho[idx + nx];
        nb[4] = rho[idx - D.nxy];
        nb[5] = rho[idx + D.nxy];
      }
      auto in_double = [&]() -> T {
        if (printed) return (T)(S.c * (double)rc);
        double lap = -6.0 * (double)rc;
#pragma unroll
        for (int q = 0; q < 6; q++) lap += (double)nb[q];
        return (T)(S.c * ((double)rc + lap / 12.0));
      };
      T v;
      if constexpr (PAIRS) {
        if (printed) {
          v = fmaf(rc, S.ch, rc * S.cl);
        } else {
          // c / 12 (6 rho + sum), the products to 2^-46
          SourcePair s = {6.0f * rc, 0.0f};
          s.lo = fmaf(6.0f, rc, -s.hi);
#pragma unroll
          for (int q = 0; q < 6; q++) pair_add(s, nb[q]);
          const float p = s.hi * S.c12h;
          v = p + (fmaf(s.hi, S.c12h, -p) + fmaf(s.hi, S.c12l, s.lo * S.c12h));
        }
        if (!(fabsf(v) <= FLT_MAX)) v = in_double();
      } else {
        v = in_double();
      }
      out[idx] = v;
    }
  }
}

// The cells of the grid's boundary, a thread each (inside the rows of rhs_kernel they would
// hold up warps of interior cells; 128^3 FP32: 125 us then, 9 + 13 apart): the source as above
// with rho = 0 outside, in FP64, minus the stencil weights times the shell values next to the
// cell.
__host__ __device__ __forceinline__ long long edge_cells(const Dims& D) {
  const long long nx = D.n[0], ny = D.n[1], nz = D.n[2];
  const long long in_x = nx > 2 ? nx - 2 : 0, in_y = ny > 2 ? ny - 2 : 0, in_z = nz > 2 ? nz - 2 : 0;
  return nx * ny * nz - in_x * in_y * in_z;
}
template <typename T>
__global__ void __launch_bounds__(kThreads) rhs_edge_kernel(const T* __restrict__ rho,
                                                            T* __restrict__ out, Dims D, double h,
                                                            double G,
                                                            const double* __restrict__ shell,
                                                            int printed) {
  const double c = 4.0 * M_PI * G * h * h;
  const int nx = D.n[0], ny = D.n[1], nz = D.n[2];
  const long long n = edge_cells(D);
  const long long planes = (long long)(nz > 1 ? 2 : 1) * D.nxy;  // whole boundary planes first
  const int per_rows = (ny > 1 ? 2 : 1) * nx, per = per_rows + (ny > 2 ? ny - 2 : 0) * (nx > 1 ? 2 : 1);
  for (long long q = (long long)blockIdx.x * kThreads + threadIdx.x; q < n;
       q += (long long)gridDim.x * kThreads) {
    int i, j, k;
    if (q < planes) {
      k = q < D.nxy ? 0 : nz - 1;
      j = (int)(q % D.nxy) / nx;
      i = (int)(q % D.nxy) % nx;
    } else {
      const long long r = q - planes;
      k = 1 + (int)(r / per);
      const int e = (int)(r % per);
      if (e < per_rows) {
        j = e < nx ? 0 : ny - 1;
        i = e % nx;
      } else {
        const int d = e - per_rows;
        i = d < ny - 2 ? 0 : nx - 1;
        j = 1 + d % (ny - 2);
      }
    }
    const long long idx = (long long)k * D.nxy + (long long)j * nx + i;
    const double rc = (double)rho[idx];
    double src = rc;
    if (!printed) {
      double lap = -6.0 * rc;
      if (i > 0) lap += (double)rho[idx - 1];
      if (i < nx - 1) lap += (double)rho[idx + 1];
      if (j > 0) lap += (double)rho[idx - nx];
      if (j < ny - 1) lap += (double)rho[idx + nx];
      if (k > 0) lap += (double)rho[idx - D.nxy];
      if (k < nz - 1) lap += (double)rho[idx + D.nxy];
      src = rc + lap / 12.0;
    }
    double v = c * src;
    for (int dz = -1; dz <= 1; dz++)
      for (int dy = -1; dy <= 1; dy++) {
        const bool out_yz = j + dy < 0 || j + dy >= ny || k + dz < 0 || k + dz >= nz;
        for (int dx = -1; dx <= 1; dx++) {
          const int ii = i + dx;
          if (!out_yz && ii >= 0 && ii < nx) continue;
          const int nnz = (dx != 0) + (dy != 0) + (dz != 0);
          const double w = nnz == 1 ? 4.0 / 9.0 : (nnz == 2 ? 1.0 / 9.0 : 1.0 / 36.0);
          v -= w * shell[shell_at(D, ii, j + dy, k + dz)];
        }
      }
    out[idx] = (T)v;
  }
}

// Odd extension of every line along `axis` to M = 2 (N + 1) points:
// (0, w_0 .. w_{N-1}, 0, -w_{N-1} .. -w_0).  Layout of the extension: axis 0 line-major
// (line * M + p); axes 1 and 2 position-major (p * B + b), b the line's index over the
// other two axes in memory order, so both the reads and the stores are coalesced.  A thread
// stores the two images of each of its cells, those of a line's ends also the zeros before them.
template <typename T, bool WARP>
__global__ void __launch_bounds__(kThreads) dst_pack_kernel(const T* __restrict__ w, T* __restrict__ ext,
                                                            Dims D, RowPieces R, int axis) {
  const int N = D.n[axis], nx = D.n[0], M = 2 * (N + 1);
  const long long B = D.ncell / N;
  const RowWalk<WARP> W(R);
  for (unsigned r = W.first; r < R.items; r += W.groups) {
    const RowItem t = row_item(D, R, r, W.lane);
    const T* const src = w + t.row * nx;
    if (axis == 0) {
      T* const line = ext + t.row * M;
      for (int i0 = t.i0; i0 < t.i1; i0 += kBatch * W.step) {
        T v[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; u++)
          if (i0 + u * W.step < t.i1) v[u] = src[i0 + u * W.step];
#pragma unroll
        for (int u = 0; u < kBatch; u++) {
          const int i = i0 + u * W.step;
          if (i < t.i1) {
            line[i + 1] = v[u];
            line[M - 1 - i] = -v[u];
          }
        }
      }
      if (t.i0 == 0) line[0] = line[N + 1] = T(0);
    } else {
      const int q = axis == 1 ? t.j : t.k;  // position along the axis
      T* const lines = ext + (long long)(axis == 1 ? t.k : t.j) * nx;
      T* const dst = lines + (q + 1) * B;
      T* const image = lines + (M - 1 - q) * B;
      for (int i0 = t.i0; i0 < t.i1; i0 += kBatch * W.step) {
        T v[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; u++)
          if (i0 + u * W.step < t.i1) v[u] = src[i0 + u * W.step];
#pragma unroll
        for (int u = 0; u < kBatch; u++) {
          const int i = i0 + u * W.step;
          if (i < t.i1) {
            dst[i] = v[u];
            image[i] = -v[u];
          }
        }
      }
      if (q == 0)
        for (int i = t.i0; i < t.i1; i += W.step) lines[i] = T(0);
      if (q == N - 1)
        for (int i = t.i0; i < t.i1; i += W.step) lines[(N + 1) * B + i] = T(0);
    }
  }
}

// Sine amplitudes back into the work array: S_k = -Im(Y_k) / 2, k = q + 1 (the halving is
// exact).  `tab` non-NULL (the last axis of the forward transform): also divided by the
// eigenvalue 6 (prod - 1), with the inverse transform's scale folded in: times
// c / (1 - tz ty tx), c = -scale / 6 (a table value, as tab's).
template <typename T, bool WARP>
__global__ void __launch_bounds__(kThreads) dst_unpack_kernel(const T* __restrict__ spec,
                                                              T* __restrict__ w, Dims D,
                                                              RowPieces R, int axis,
                                                              const double* __restrict__ tab,
                                                              double coef) {
  using V = typename TableOf<T>::type;
  const V* const tx = reinterpret_cast<const V*>(tab);
  const V* const ty = tx + D.n[0];
  const V* const tz = ty + D.n[1];
  const V c = *reinterpret_cast<const V*>(&coef);
  const int nx = D.n[0], N = D.n[axis];
  const long long B = D.ncell / N;
  const long long half = N + 2;  // M / 2 + 1 complex values per line
  const RowWalk<WARP> W(R);
  for (unsigned q = W.first; q < R.items; q += W.groups) {
    const RowItem t = row_item(D, R, q, W.lane);
    const long long ci = axis == 0 ? t.row * half + 1
                                   : (axis == 1 ? (long long)(t.j + 1) * B + (long long)t.k * nx
                                                : (long long)(t.k + 1) * B + (long long)t.j * nx);
    V tzy = V();
    if (tab) tzy = table_product(tz[t.k], ty[t.j]);
    for (int i0 = t.i0; i0 < t.i1; i0 += kBatch * W.step) {
      T v[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; u++)
        if (i0 + u * W.step < t.i1) v[u] = T(-0.5) * spec[2 * (ci + i0 + u * W.step) + 1];
#pragma unroll
      for (int u = 0; u < kBatch; u++) {
        const int i = i0 + u * W.step;
        if (i >= t.i1) break;
        if (tab) v[u] = scaled(v[u], over_one_minus(c, tzy, tx[i]));
        w[t.row * nx + i] = v[u];
      }
    }
  }
}

// ---------------------------------------------------- dense sine transforms (FP32)
// A type-I sine transform along one axis of N <= kDenseMax points as a matrix product.  The
// symmetry sin(pi j (N - i) / (N + 1)) = -+ sin(pi j (i + 1) / (N + 1)) halves it: the odd
// j take the sums w_i + w_{N-1-i}, the even j the differences.  A CTA holds 64 lines and the
// matrix in shared memory; a warp forms 16 outputs of one parity for two columns per lane,
// on packed FMAs, in chains of four terms, two of which are added before they join the sum: the
// rounding of the sums is what the solve's error is made of.  Against 64 bits (relative L2, mean
// of six blobs) 47^3 1.57e-7, 53^3 1.51e-7, 64 x 64 x 40 1.36e-7, where the transform of the odd
// extension has 1.57e-7, 1.72e-7 and 1.72e-7, and chains of sixteen 1.96e-7, 1.94e-7 and 1.95e-7
// (2 % faster); on most larger sizes the fast transform has twice the error.
// 128^3: 134 M FMAs a transform, 3.4 us at the FMA peak, beside 16.8 MB of traffic; the odd
// extension, the real transform of 2 (N + 1) points and the unpacking took about 100 us each
// (258 = 2 3 43 is a poor length), the six transforms of a solve take 105 so.
// N^2 work: beyond kDenseMax the matrix does not fit and the transform of the extension is used.
constexpr int kDenseMax = 256;
constexpr int kDenseCols = 64;
constexpr int kDenseOut = 16;

// The matrix in the order the warps read it: chunks of 16 outputs (first those of odd j, then
// of even j), each [term][16], zero beyond the last output.
struct DenseDims {
  int N, terms[2], outs[2], chunks[2];
};
__host__ __device__ inline DenseDims dense_dims(int N) {
  DenseDims d;
  d.N = N;
  d.terms[0] = d.outs[0] = (N + 1) / 2;
  d.terms[1] = d.outs[1] = N / 2;
  for (int q = 0; q < 2; q++) d.chunks[q] = (d.outs[q] + kDenseOut - 1) / kDenseOut;
  return d;
}
__host__ __device__ inline int dense_matrix(const DenseDims& d) {
  return kDenseOut * (d.chunks[0] * d.terms[0] + d.chunks[1] * d.terms[1]);
}
size_t dense_smem(int N) {
  return sizeof(float) * ((size_t)dense_matrix(dense_dims(N)) + (size_t)N * kDenseCols);
}

// The transform of the 64 lines in D (D[i][column]), in place; matrix in Sm.  Barriers around.
__device__ __forceinline__ void dense_sine(float* D, const float* Sm, const DenseDims& d) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int N = d.N, h = d.terms[1];
  // sums to the first half, differences to the mirrored places (the middle one stays)
  for (int e = threadIdx.x; e < h * kDenseCols; e += kThreads) {
    const int i = e / kDenseCols, c = e % kDenseCols;
    const float x = D[i * kDenseCols + c], y = D[(N - 1 - i) * kDenseCols + c];
    D[i * kDenseCols + c] = x + y;
    D[(N - 1 - i) * kDenseCols + c] = x - y;
  }
  __syncthreads();
  // each warp's outputs stay in registers until every warp has read D
  constexpr int kMaxChunks = (kDenseMax / kDenseOut + kThreads / 32 - 1) / (kThreads / 32);
  float2 out[kMaxChunks][kDenseOut / 2][2];
  const int chunks = d.chunks[0] + d.chunks[1];
#pragma unroll
  for (int r = 0; r < kMaxChunks; r++) {
    const int ch = warp + r * (kThreads / 32);
#pragma unroll
    for (int q = 0; q < kDenseOut / 2; q++) out[r][q][0] = out[r][q][1] = make_float2(0.0f, 0.0f);
    if (ch >= chunks) continue;
    const bool odd = ch < d.chunks[0];
    const int terms = d.terms[odd ? 0 : 1];
    const float* m = Sm + kDenseOut * (odd ? ch * d.terms[0]
                                           : d.chunks[0] * d.terms[0] +
                                                 (ch - d.chunks[0]) * d.terms[1]);
    const float* x = D + (odd ? 0 : (N - 1) * kDenseCols) + lane;
    const int step = odd ? kDenseCols : -kDenseCols;
    // eight terms (n of them at the end) of half of the outputs at a time: two chains of four,
    // their sum added to the outputs
    auto group = [&](int i0, auto full, int n) {
      constexpr bool FULL = decltype(full)::value;
#pragma unroll
      for (int half = 0; half < 2; half++) {
        float2 sum[2][kDenseOut / 4][2];
#pragma unroll
        for (int c = 0; c < 2; c++)
#pragma unroll
          for (int t = 0; t < 4; t++) {
            const int i = i0 + 4 * c + t;
            if (!FULL && 4 * c + t >= n) {
              if (t > 0) break;
#pragma unroll
              for (int q = 0; q < kDenseOut / 4; q++) sum[c][q][0] = sum[c][q][1] = both(0.0f);
              break;
            }
            const float2 a = both(x[i * step]), b = both(x[i * step + 32]);
            const float4* row = reinterpret_cast<const float4*>(m + i * kDenseOut) + 2 * half;
#pragma unroll
            for (int q = 0; q < kDenseOut / 8; q++) {
              const float4 w = row[q];
              const float2 w0 = make_float2(w.x, w.y), w1 = make_float2(w.z, w.w);
              float2(*const s0)[2] = &sum[c][2 * q];
              s0[0][0] = t == 0 ? mul2(w0, a) : fma2(w0, a, s0[0][0]);
              s0[0][1] = t == 0 ? mul2(w0, b) : fma2(w0, b, s0[0][1]);
              s0[1][0] = t == 0 ? mul2(w1, a) : fma2(w1, a, s0[1][0]);
              s0[1][1] = t == 0 ? mul2(w1, b) : fma2(w1, b, s0[1][1]);
            }
          }
#pragma unroll
        for (int q = 0; q < kDenseOut / 4; q++)
#pragma unroll
          for (int k = 0; k < 2; k++) {
            float2& o = out[r][half * (kDenseOut / 4) + q][k];
            o = add2(o, add2(sum[0][q][k], sum[1][q][k]));
          }
      }
    };
    int i0 = 0;
    for (; i0 + 8 <= terms; i0 += 8) group(i0, std::true_type(), 8);
    if (i0 < terms) group(i0, std::false_type(), terms - i0);
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kMaxChunks; r++) {
    const int ch = warp + r * (kThreads / 32);
    if (ch >= chunks) continue;
    const bool odd = ch < d.chunks[0];
    const int o0 = kDenseOut * (odd ? ch : ch - d.chunks[0]), outs = d.outs[odd ? 0 : 1];
#pragma unroll
    for (int q = 0; q < kDenseOut; q++) {
      if (o0 + q >= outs) break;
      float* row = D + (2 * (o0 + q) + (odd ? 0 : 1)) * kDenseCols + lane;  // output j - 1
      row[0] = q & 1 ? out[r][q / 2][0].y : out[r][q / 2][0].x;
      row[32] = q & 1 ? out[r][q / 2][1].y : out[r][q / 2][1].x;
    }
  }
  __syncthreads();
}

// The lines along `axis`, 64 per CTA, transformed in place.  tab non-NULL (axis 2 only): the
// amplitudes are divided by the operator's eigenvalue (see dst_unpack_kernel) and transformed
// back at once.
__global__ void __launch_bounds__(kThreads, 2) dense_sine_kernel(float* __restrict__ w,
                                                              const float* __restrict__ matrix,
                                                              Dims D, int axis,
                                                              const double* __restrict__ tab,
                                                              double coef) {
  extern __shared__ __align__(16) float dense_mem[];
  const DenseDims d = dense_dims(D.n[axis]);
  const int nm = dense_matrix(d), N = d.N;
  float* const Sm = dense_mem;
  float* const X = dense_mem + nm;
  const long long lines = D.ncell / N, l0 = (long long)blockIdx.x * kDenseCols;
  for (int e = threadIdx.x; e < nm / 4; e += kThreads)
    reinterpret_cast<float4*>(Sm)[e] = reinterpret_cast<const float4*>(matrix)[e];
  const int cols = (int)(lines - l0 < kDenseCols ? lines - l0 : kDenseCols);
  // axis 0: a warp reads lines of consecutive values; else threads take consecutive lines
  const long long stride = axis == 1 ? D.n[0] : D.nxy;
  const int col = threadIdx.x % kDenseCols;
  const long long line = l0 + col;
  const long long base = axis == 1 ? line / D.n[0] * D.nxy + line % D.n[0] : line;
  auto each = [&](auto op) {
    if (axis == 0) {
      for (int c = threadIdx.x / 32; c < kDenseCols; c += kThreads / 32)
        for (int i = threadIdx.x & 31; i < N; i += 32)
          op(i, c, (l0 + c) * N + i, c < cols);
    } else {
      for (int i = threadIdx.x / kDenseCols; i < N; i += kThreads / kDenseCols)
        op(i, col, base + i * stride, col < cols);
    }
  };
  each([&](int i, int c, long long o, bool ok) { X[i * kDenseCols + c] = ok ? w[o] : 0.0f; });
  __syncthreads();
  dense_sine(X, Sm, d);
  if (tab) {
    const FloatPair* const tx = reinterpret_cast<const FloatPair*>(tab);
    const FloatPair* const ty = tx + D.n[0];
    const FloatPair* const tz = ty + D.n[1];
    const FloatPair cf = *reinterpret_cast<const FloatPair*>(&coef);
    if (col < cols) {
      const FloatPair txy = table_product(ty[line / D.n[0]], tx[line % D.n[0]]);
      for (int i = threadIdx.x / kDenseCols; i < N; i += kThreads / kDenseCols)
        X[i * kDenseCols + col] = scaled(X[i * kDenseCols + col], over_one_minus(cf, txy, tz[i]));
    }
    __syncthreads();
    dense_sine(X, Sm, d);
  }
  each([&](int i, int c, long long o, bool ok) {
    if (ok) w[o] = X[i * kDenseCols + c];
  });
}

int blocks_for(long long n) {
  const long long b = (n + kThreads - 1) / kThreads;
  return (int)(b < 152LL * 16 ? (b > 0 ? b : 1) : 152LL * 16);
}

}  // namespace

struct PoissonIso {
  int n[3];
  int dtype;
  cufftHandle plan[3];
  int nplans;
  void* ext;
  void* spec;
  double* part;
  double* mom;
  double* tab;
  double* shell;  // the potential on the cells around the grid
  float* sine[3];  // FP32 grids of at most kDenseMax points per axis: the sine matrices
};

void ppml_iso_free(PoissonIso* s) {
  if (!s) return;
  for (int a = 0; a < s->nplans; a++) cufftDestroy(s->plan[a]);
  if (s->ext) cudaFree(s->ext);
  if (s->spec) cudaFree(s->spec);
  if (s->part) cudaFree(s->part);
  if (s->mom) cudaFree(s->mom);
  if (s->tab) cudaFree(s->tab);
  if (s->shell) cudaFree(s->shell);
  for (int a = 0; a < 3; a++)
    if (s->sine[a]) cudaFree(s->sine[a]);
  delete s;
}

static int iso_create(const ppml_grid_desc* d, PoissonIso** out) {
  PoissonIso* s = new PoissonIso();
  s->n[0] = d->nx;
  s->n[1] = d->ny;
  s->n[2] = d->nz;
  s->dtype = d->dtype;
  const bool f64 = d->dtype == PPML_F64;
  const size_t elt = f64 ? sizeof(double) : sizeof(float);
  const long long ncell = (long long)d->nx * d->ny * d->nz;
  Dims D;
  for (int a = 0; a < 3; a++) D.n[a] = s->n[a];
  size_t ext_n = 0, spec_n = 0;
  for (int a = 0; a < 3; a++) {
    const long long N = s->n[a], B = ncell / N;
    if ((size_t)(2 * (N + 1) * B) > ext_n) ext_n = (size_t)(2 * (N + 1) * B);
    if ((size_t)((N + 2) * B) > spec_n) spec_n = (size_t)((N + 2) * B);
  }
  bool dense = !f64;
  for (int a = 0; a < 3; a++) dense = dense && s->n[a] <= kDenseMax;
  if (dense) ext_n = spec_n = 0;
  if ((ext_n && cudaMalloc(&s->ext, ext_n * elt) != cudaSuccess) ||
      (spec_n && cudaMalloc(&s->spec, spec_n * 2 * elt) != cudaSuccess) ||
      cudaMalloc(&s->part, sizeof(double) * kMoments * kMaxMomentBlocks) != cudaSuccess ||
      cudaMalloc(&s->mom, sizeof(double) * kMoments) != cudaSuccess ||
      cudaMalloc(&s->tab, sizeof(double) * (size_t)(s->n[0] + s->n[1] + s->n[2])) != cudaSuccess ||
      cudaMalloc(&s->shell, sizeof(double) * (size_t)shell_cells(D)) != cudaSuccess) {
    cudaGetLastError();
    ppml_iso_free(s);
    return ppml_fail(PPML_E_NOMEM, "isolated Poisson buffers (%zu + %zu elements)", ext_n,
                     2 * spec_n);
  }
  std::vector<double> tab;
  for (int a = 0; a < 3; a++)
    for (int q = 0; q < s->n[a]; q++) {
      const double sn = sin(M_PI * (double)(q + 1) / (2.0 * (double)(s->n[a] + 1)));
      tab.push_back(ppml_table_value(1.0 - (2.0 / 3.0) * sn * sn, f64));
    }
  if (cudaMemcpy(s->tab, tab.data(), sizeof(double) * tab.size(), cudaMemcpyHostToDevice) !=
      cudaSuccess) {
    ppml_iso_free(s);
    return ppml_fail(PPML_E_CUDA, "isolated Poisson tables: %s",
                     cudaGetErrorString(cudaGetLastError()));
  }
  for (int a = 0; a < 3 && dense; a++) {
    const DenseDims d = dense_dims(s->n[a]);
    std::vector<float> m((size_t)dense_matrix(d), 0.0f);
    float* at = m.data();
    for (int q = 0; q < 2; q++)
      for (int ch = 0; ch < d.chunks[q]; ch++)
        for (int i = 0; i < d.terms[q]; i++)
          for (int o = 0; o < kDenseOut; o++, at++) {
            const int k = ch * kDenseOut + o;  // output of this parity: j = 2 k + 1 + q
            if (k < d.outs[q])
              *at = (float)sin(M_PI * (double)((long long)(2 * k + 1 + q) * (i + 1) % (2LL * (d.N + 1))) /
                               (double)(d.N + 1));
          }
    if (cudaMalloc(&s->sine[a], sizeof(float) * m.size()) != cudaSuccess) {
      cudaGetLastError();
      ppml_iso_free(s);
      return ppml_fail(PPML_E_NOMEM, "isolated Poisson sine matrix (%zu elements)", m.size());
    }
    cudaError_t e = cudaMemcpy(s->sine[a], m.data(), sizeof(float) * m.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(dense_sine_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)dense_smem(kDenseMax));
    if (e != cudaSuccess) {
      ppml_iso_free(s);
      return ppml_fail(PPML_E_CUDA, "isolated Poisson sine matrix: %s", cudaGetErrorString(e));
    }
  }
  for (int a = 0; a < 3 && !dense; a++) {
    int M = 2 * (s->n[a] + 1);
    int inembed[1] = {M}, onembed[1] = {M / 2 + 1};
    const int B = (int)(ncell / s->n[a]);
    const int istride = a == 0 ? 1 : B, idist = a == 0 ? M : 1;
    const int ostride = a == 0 ? 1 : B, odist = a == 0 ? M / 2 + 1 : 1;
    if (cufftPlanMany(&s->plan[a], 1, &M, inembed, istride, idist, onembed, ostride, odist,
                      f64 ? CUFFT_D2Z : CUFFT_R2C, B) != CUFFT_SUCCESS) {
      ppml_iso_free(s);
      return ppml_fail(PPML_E_CUDA, "cufftPlanMany for the sine transform along axis %d", a);
    }
    s->nplans = a + 1;
  }
  *out = s;
  return PPML_OK;
}

template <typename T, bool WARP>
static int iso_run(PoissonIso* s, const T* rho, T* phi, double h, double G, int printed,
                   cudaStream_t st) {
  Dims D;
  for (int a = 0; a < 3; a++) D.n[a] = s->n[a];
  D.nxy = (long long)D.n[0] * D.n[1];
  D.ncell = D.nxy * D.n[2];
  int blocks;
  const long long rows = D.ncell / D.n[0];
  if (sizeof(T) == sizeof(float) && D.n[0] <= kPairMax && D.n[1] <= kPairMax &&
      (D.nxy >= kPairPlane || D.n[2] <= kMaxMomentBlocks)) {
    const int most = (int)std::max(1LL, std::min<long long>(D.nxy / kPairItem, D.n[1]));
    const int cuts = std::min((kPairBlocks + D.n[2] - 1) / D.n[2], most);
    blocks = (int)std::min<long long>((long long)D.n[2] * cuts, kMaxMomentBlocks);
    moment_pair_kernel<<<blocks, kThreads, 0, st>>>(
        (const float*)rho, D, row_pieces(D.n[0], D.n[1], (D.n[1] + cuts - 1) / cuts, kThreads, 8), cuts,
        IndexDivisor(cuts), h, s->part);
  } else {
    blocks = std::min(blocks_for(D.ncell), kMaxMomentBlocks);
    moment_kernel<T, WARP><<<blocks, kThreads, 0, st>>>(
        rho, D, row_pieces(D.n[0], D.n[1], rows, (long long)blocks * kThreads, 8), h, s->part);
  }
  int rc = ppml_check_launch("moment_kernel");
  if (rc) return rc;
  moment_final_kernel<<<1, kThreads, 0, st>>>(s->part, blocks, s->mom);
  if ((rc = ppml_check_launch("moment_final_kernel"))) return rc;
  shell_kernel<<<blocks_for(shell_cells(D)), kThreads, 0, st>>>(D, h, G, s->mom, s->shell);
  if ((rc = ppml_check_launch("shell_kernel"))) return rc;
  const Source source(4.0 * M_PI * G * h * h);
  const RowPieces R = row_pieces(D.n[0], D.n[1], rows, (long long)blocks_for(D.ncell) * kThreads, 1);
  if (sizeof(T) == sizeof(float) && ppml_pair_range(source.c, 1.0) && ppml_pair_range(source.c / 12.0, 1.0))
    rhs_kernel<float, true, WARP><<<blocks_for(D.ncell), kThreads, 0, st>>>((const float*)rho, (float*)phi,
                                                                      D, R, source, printed);
  else
    rhs_kernel<T, false, WARP><<<blocks_for(D.ncell), kThreads, 0, st>>>(rho, phi, D, R, source, printed);
  if ((rc = ppml_check_launch("rhs_kernel"))) return rc;
  rhs_edge_kernel<T><<<blocks_for(edge_cells(D)), kThreads, 0, st>>>(rho, phi, D, h, G, s->shell,
                                                                     printed);
  if ((rc = ppml_check_launch("rhs_kernel"))) return rc;
  double scale = 1.0;
  for (int a = 0; a < 3; a++) scale *= 2.0 / (double)(D.n[a] + 1);
  const double symbol = ppml_table_value(-scale / 6.0, sizeof(T) == sizeof(double));
  if constexpr (sizeof(T) == sizeof(float)) {
    if (s->sine[0]) {  // x, y, then z there and back, y, x
      const int order[5] = {0, 1, 2, 1, 0};
      for (int q = 0; q < 5; q++) {
        const int a = order[q];
        const long long lines = D.ncell / D.n[a];
        dense_sine_kernel<<<(int)((lines + kDenseCols - 1) / kDenseCols), kThreads,
                            dense_smem(D.n[a]), st>>>(phi, s->sine[a], D, a,
                                                      q == 2 ? s->tab : nullptr, symbol);
        if ((rc = ppml_check_launch("dense_sine_kernel"))) return rc;
      }
      return PPML_OK;
    }
  }
  for (int pass = 0; pass < 2; pass++) {
    for (int a = 0; a < 3; a++) {
      dst_pack_kernel<T, WARP><<<blocks_for(D.ncell), kThreads, 0, st>>>(phi, (T*)s->ext, D, R, a);
      if ((rc = ppml_check_launch("dst_pack_kernel"))) return rc;
      if (cufftSetStream(s->plan[a], st) != CUFFT_SUCCESS)
        return ppml_fail(PPML_E_CUDA, "cufftSetStream failed");
      cufftResult r;
      if (sizeof(T) == sizeof(double))
        r = cufftExecD2Z(s->plan[a], (cufftDoubleReal*)s->ext, (cufftDoubleComplex*)s->spec);
      else
        r = cufftExecR2C(s->plan[a], (cufftReal*)s->ext, (cufftComplex*)s->spec);
      if (r != CUFFT_SUCCESS) return ppml_fail(PPML_E_CUDA, "cuFFT sine transform failed (%d)", (int)r);
      dst_unpack_kernel<T, WARP><<<blocks_for(D.ncell), kThreads, 0, st>>>(
          (const T*)s->spec, phi, D, R, a, pass == 0 && a == 2 ? s->tab : nullptr, symbol);
      if ((rc = ppml_check_launch("dst_unpack_kernel"))) return rc;
    }
  }
  return PPML_OK;
}

int ppml_iso_solve(PoissonIso** state, const ppml_grid_desc* d, const void* rho, void* phi,
                   double G, unsigned flags, cudaStream_t st) {
  if (!*state) {
    int rc = iso_create(d, state);
    if (rc) return rc;
  }
  PoissonIso* s = *state;
  const int printed = (flags & PPML_POISSON_PRINTED_RHS) != 0;
  auto run = [&](auto warp) {
    constexpr bool W = decltype(warp)::value;
    if (d->dtype == PPML_F64)
      return iso_run<double, W>(s, (const double*)rho, (double*)phi, d->h[0], G, printed, st);
    return iso_run<float, W>(s, (const float*)rho, (float*)phi, d->h[0], G, printed, st);
  };
  // rows of at least a warp's half have a warp each, shorter ones share it
  return s->n[0] > 16 ? run(std::true_type()) : run(std::false_type());
}
