// Definitions of the launchers for one precision PPML_REAL (included by
// ppml_kern_f32.cu / ppml_kern_f64.cu).
#include <algorithm>

#include "../../include/ppml.h"
#include "ppml_internal.h"
#include "ppml_launch.h"
#include "ppml_thin.cuh"

namespace ppml {

// Kernels of their own for plain float states (ppml_kern_f32.cu); FP64 has none.
inline bool launch_euler_sweeps(const MarchArgs<double>&, int, cudaStream_t) { return false; }
inline bool launch_sweeps(const MarchArgs<double>&, int, cudaStream_t) { return false; }
inline cudaError_t prepare_sweeps(double) { return cudaSuccess; }

namespace {
// CTAs per SM the march kernels are compiled for (register budget per thread)
template <typename T>
struct MinBlocks;
template <>
struct MinBlocks<float> {
  static constexpr int value = 2;
};
template <>
struct MinBlocks<double> {
  static constexpr int value = 1;
};
}  // namespace

// Double-float states (low parts of rho, m, rho E) exist only in the FP32 path.
constexpr bool kHasDF = sizeof(PPML_REAL) == 4;

template <bool DF, bool INF>
cudaError_t set_stage_smem_one() {
  constexpr int MB = MinBlocks<PPML_REAL>::value;
  cudaError_t e = cudaFuncSetAttribute(lagrangian_tile<PPML_REAL, MB, DF, INF>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(LagTileSmem<PPML_REAL>));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(eulerian_tile<PPML_REAL, MB, DF, INF>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(EulTileSmem<PPML_REAL>));
  return e;
}
template <bool DF>
cudaError_t set_stage_smem() {
  cudaError_t e = set_stage_smem_one<DF, false>();
  if (e == cudaSuccess) e = set_stage_smem_one<DF, true>();
  return e;
}

namespace {
// Grids with one or two active axes, plain states (ppml_thin.cuh).
template <bool FLAT, bool TWO>
void launch_thin_eulerian(const MarchArgs<PPML_REAL>& A, cudaStream_t st) {
  ThinGeom t;
  const int n = thin_tiles<ThinShape<PPML_REAL, TWO>>(A.g, t);
  if constexpr (sizeof(PPML_REAL) == 8 && !TWO)
    thin1d_eulerian_f64<FLAT><<<n, THIN_NT, 0, st>>>(A);
  else
    thin_eulerian<PPML_REAL, FLAT, TWO><<<n, THIN_NT, 0, st>>>(A);
}
template <bool FLAT, bool TWO>
void launch_thin_lagrangian(const MarchArgs<PPML_REAL>& A, cudaStream_t st) {
  using S = ThinShape<PPML_REAL, TWO>;
  ThinGeom t;
  const int n = thin_tiles<S>(A.g, t);
  if constexpr (sizeof(PPML_REAL) == 8 && !TWO)
    thin1d_lagrangian_f64<FLAT><<<n, THIN_NT, 0, st>>>(A);
  else
    thin_lagrangian<PPML_REAL, FLAT, TWO>
        <<<n, THIN_NT, sizeof(ThinLagSmem<PPML_REAL, S>), st>>>(A);
}
template <bool FLAT, bool TWO>
cudaError_t prepare_thin() {
  if constexpr (sizeof(PPML_REAL) == 8 && !TWO)
    return cudaSuccess;
  else
    return cudaFuncSetAttribute(thin_lagrangian<PPML_REAL, FLAT, TWO>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sizeof(ThinLagSmem<PPML_REAL, ThinShape<PPML_REAL, TWO>>));
}
bool launch_thin(const MarchArgs<PPML_REAL>& A, bool eulerian, cudaStream_t st) {
  if (!thin_grid(A.g) || (eulerian && A.phi)) return false;
  const bool flat = (A.flags & PPML_FIRST_ORDER) != 0, two = thin_axes(A.g).axB >= 0;
  if (eulerian) {
    if (flat)
      two ? launch_thin_eulerian<true, true>(A, st) : launch_thin_eulerian<true, false>(A, st);
    else
      two ? launch_thin_eulerian<false, true>(A, st) : launch_thin_eulerian<false, false>(A, st);
  } else {
    if (flat)
      two ? launch_thin_lagrangian<true, true>(A, st) : launch_thin_lagrangian<true, false>(A, st);
    else
      two ? launch_thin_lagrangian<false, true>(A, st) : launch_thin_lagrangian<false, false>(A, st);
  }
  return true;
}
}  // namespace

template <>
int prepare_kernels<PPML_REAL>() {
  cudaError_t e = set_stage_smem<false>();
  if (e == cudaSuccess) e = prepare_sweeps(PPML_REAL(0));
  if (e == cudaSuccess) e = prepare_thin<false, false>();
  if (e == cudaSuccess) e = prepare_thin<false, true>();
  if (e == cudaSuccess) e = prepare_thin<true, false>();
  if (e == cudaSuccess) e = prepare_thin<true, true>();
  if (e == cudaSuccess && kHasDF) e = set_stage_smem<kHasDF>();
  if (e != cudaSuccess) return ppml_fail(PPML_E_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
  return PPML_OK;
}

template <>
int launch_eulerian<PPML_REAL>(const MarchArgs<PPML_REAL>& A, int nblk, cudaStream_t st) {
  constexpr int MB = MinBlocks<PPML_REAL>::value;
  constexpr size_t SM = sizeof(EulTileSmem<PPML_REAL>);
  const bool df = kHasDF && A.outlo[1];
  if (!df && launch_thin(A, true, st)) return ppml_check_launch("thin_eulerian");
  if (!df && launch_euler_sweeps(A, nblk, st)) return ppml_check_launch("eulerian_sweep_f32");
  if (A.any_inflow) {
    if (df)
      eulerian_tile<PPML_REAL, MB, kHasDF, true><<<nblk, TN, SM, st>>>(A);
    else
      eulerian_tile<PPML_REAL, MB, false, true><<<nblk, TN, SM, st>>>(A);
  } else if (df) {
    eulerian_tile<PPML_REAL, MB, kHasDF, false><<<nblk, TN, SM, st>>>(A);
  } else {
    eulerian_tile<PPML_REAL, MB, false, false><<<nblk, TN, SM, st>>>(A);
  }
  return ppml_check_launch("eulerian_tile");
}

template <>
int launch_lagrangian<PPML_REAL>(const MarchArgs<PPML_REAL>& A, int nblk, cudaStream_t st) {
  constexpr int MB = MinBlocks<PPML_REAL>::value;
  constexpr size_t SM = sizeof(LagTileSmem<PPML_REAL>);
  const bool df = kHasDF && A.outlo[0];
  if (!df && launch_thin(A, false, st)) return ppml_check_launch("thin_lagrangian");
  if (!df && launch_sweeps(A, nblk, st)) return ppml_check_launch("lagrangian_sweep_f32");
  if (A.any_inflow) {
    if (df)
      lagrangian_tile<PPML_REAL, MB, kHasDF, true><<<nblk, TN, SM, st>>>(A);
    else
      lagrangian_tile<PPML_REAL, MB, false, true><<<nblk, TN, SM, st>>>(A);
  } else if (df) {
    lagrangian_tile<PPML_REAL, MB, kHasDF, false><<<nblk, TN, SM, st>>>(A);
  } else {
    lagrangian_tile<PPML_REAL, MB, false, false><<<nblk, TN, SM, st>>>(A);
  }
  return ppml_check_launch("lagrangian_tile");
}

template <>
int launch_diag<PPML_REAL>(const MarchArgs<PPML_REAL>& A, int nblk, cudaStream_t st) {
  diag_kernel<PPML_REAL><<<nblk, NT, 0, st>>>(A);
  return ppml_check_launch("diag_kernel");
}

namespace {
// Multiply the half spectrum (R2C layout: kx in [0, nx/2], ky, kz) by the inverse symbol of
// the 27-point stencil, coef / (1 - tx ty tz); tables hold 1 - (2/3) sin^2(pi k / N) per axis
// (FP32 grids: as float pairs).  A thread per value, whatever the grid's shape (a warp per row
// of kx: 65536 x 4 x 4 in FP64 903 us, 14.6 so; 128^3, rows of 65 values, 41 and 27.5).  V: the
// arithmetic, double or (FP32 grids) float pairs, which the memory bounds: 512^3 201 us for
// 1.07 GB, 1986 with an FP64 division per value.
struct SymbolIndex {
  int mx, ny;
  unsigned n;  // values
  IndexDivisor by_mx, by_ny;
};
template <typename T, typename V>
__global__ void __launch_bounds__(256) poisson_symbol_kernel(T* spec, const double* __restrict__ tab,
                                                             SymbolIndex X, V coef) {
  using U = typename TableOf<T>::type;
  using T2 = std::conditional_t<sizeof(T) == 8, double2, float2>;
  static_assert(sizeof(U) == sizeof(double), "a table value fills a double's storage");
  T2* const s = reinterpret_cast<T2*>(spec);
  const U* const tx = reinterpret_cast<const U*>(tab);
  const U* const ty = tx + X.mx;
  const U* const tz = ty + X.ny;
  constexpr int B = sizeof(V) == sizeof(T) ? 1 : 2;  // values in flight (float pairs: memory-bound)
  const unsigned stride = gridDim.x * 256 * B;
  for (unsigned first = blockIdx.x * 256 * B + threadIdx.x; first < X.n; first += stride) {
    T2 v[B];
#pragma unroll
    for (int u = 0; u < B; u++)
      if (first + u * 256 < X.n) v[u] = s[first + u * 256];
#pragma unroll
    for (int u = 0; u < B; u++) {
      const unsigned idx = first + u * 256;
      if (idx >= X.n) break;
      const unsigned row = X.by_mx.quotient(idx), kx = idx - row * (unsigned)X.mx;
      const unsigned kz = X.by_ny.quotient(row), ky = row - kz * (unsigned)X.ny;
      const V f = over_one_minus(coef, table_product(table_as<V>(tz[kz]), table_as<V>(ty[ky])),
                                 table_as<V>(tx[kx]));
      v[u].x = scaled(v[u].x, f);
      v[u].y = scaled(v[u].y, f);
      if (idx == 0) v[u].x = v[u].y = T(0);  // the k = 0 mode
      s[idx] = v[u];
    }
  }
}

template <typename T>
void launch_symbol(T* spec, const double* tab, int mx, int ny, int nz, double coef, bool pairs,
                   cudaStream_t st) {
  const long long n = (long long)mx * ny * nz;
  const SymbolIndex X = {mx, ny, (unsigned)n, IndexDivisor(mx), IndexDivisor(ny)};
  const int blocks = (int)std::min((n + 255) / 256, 152LL * 16);
  if constexpr (sizeof(T) == 4) {
    if (pairs) {
      const float hi = (float)coef;
      const FloatPair c = {hi, (float)(coef - (double)hi)};
      poisson_symbol_kernel<T, FloatPair><<<blocks, 256, 0, st>>>(spec, tab, X, c);
      return;
    }
  }
  poisson_symbol_kernel<T, double><<<blocks, 256, 0, st>>>(spec, tab, X, coef);
}
}  // namespace

template <>
int launch_poisson_symbol<PPML_REAL>(void* spec, const double* tab, int mx, int ny, int nz,
                                     double coef, bool pairs, cudaStream_t st) {
  launch_symbol<PPML_REAL>((PPML_REAL*)spec, tab, mx, ny, nz, coef, pairs, st);
  return ppml_check_launch("poisson_symbol_kernel");
}

namespace {
// Opt-in shared memory of a kernel, raised once to the largest size launched so far.
template <typename K>
int raise_smem(K kernel, size_t smem, size_t& configured) {
  if (smem > configured) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess)
      return ppml_fail(PPML_E_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    configured = smem;
  }
  return PPML_OK;
}

template <int NT, bool DF>
int launch_batch_ntd(PPML_REAL* rho, PPML_REAL* m, PPML_REAL* en, PPML_REAL* ei,
                     BatchLo<PPML_REAL> lo, InstDev* inst, const int* order, double gamma,
                     double cfl, int max_steps, int nmax, int ninst, size_t smem,
                     cudaStream_t st) {
  static size_t configured = 0;
  int rc = raise_smem(batch_kernel<PPML_REAL, NT, DF>, smem, configured);
  if (rc) return rc;
  batch_kernel<PPML_REAL, NT, DF><<<ninst, NT, smem, st>>>(rho, m, en, ei, lo, inst, order, gamma,
                                                           cfl, max_steps, nmax);
  return ppml_check_launch("batch_kernel");
}

template <int NT, bool DF>
int launch_cluster_ntd(PPML_REAL* rho, PPML_REAL* m, PPML_REAL* en, PPML_REAL* ei,
                       BatchLo<PPML_REAL> lo, InstDev* inst, const int2* items, double gamma,
                       double cfl, int max_steps, int nlmax, int nmax, int nitems, size_t smem,
                       cudaStream_t st) {
  static size_t configured = 0;
  int rc = raise_smem(batch_cluster_kernel<PPML_REAL, NT, DF>, smem, configured);
  if (rc) return rc;
  batch_cluster_kernel<PPML_REAL, NT, DF><<<2 * nitems, NT, smem, st>>>(
      rho, m, en, ei, lo, inst, items, gamma, cfl, max_steps, nlmax, nmax);
  return ppml_check_launch("batch_cluster_kernel");
}

// double-float launches (low parts given) exist only in FP32
template <int NT>
int launch_batch_nt(PPML_REAL* rho, PPML_REAL* m, PPML_REAL* en, PPML_REAL* ei,
                    BatchLo<PPML_REAL> lo, InstDev* inst, const int* order, double gamma,
                    double cfl, int max_steps, int nmax, int ninst, size_t smem, cudaStream_t st) {
  if (kHasDF && lo.p[0])
    return launch_batch_ntd<NT, kHasDF>(rho, m, en, ei, lo, inst, order, gamma, cfl, max_steps,
                                        nmax, ninst, smem, st);
  return launch_batch_ntd<NT, false>(rho, m, en, ei, lo, inst, order, gamma, cfl, max_steps, nmax,
                                     ninst, smem, st);
}

template <int NT>
int launch_cluster_nt(PPML_REAL* rho, PPML_REAL* m, PPML_REAL* en, PPML_REAL* ei,
                      BatchLo<PPML_REAL> lo, InstDev* inst, const int2* items, double gamma,
                      double cfl, int max_steps, int nlmax, int nmax, int nitems, size_t smem,
                      cudaStream_t st) {
  if (kHasDF && lo.p[0])
    return launch_cluster_ntd<NT, kHasDF>(rho, m, en, ei, lo, inst, items, gamma, cfl, max_steps,
                                          nlmax, nmax, nitems, smem, st);
  return launch_cluster_ntd<NT, false>(rho, m, en, ei, lo, inst, items, gamma, cfl, max_steps,
                                       nlmax, nmax, nitems, smem, st);
}
}  // namespace

template <>
int launch_batch_vacuum<PPML_REAL>(const PPML_REAL* rho, InstDev* inst, int ninst,
                                   cudaStream_t st) {
  // vacuum thresholds of instances not yet started (no-op for the others)
  batch_vacuum_kernel<PPML_REAL><<<ninst, 256, 0, st>>>(rho, inst);
  return ppml_check_launch("batch_vacuum_kernel");
}

template <>
int launch_batch_cluster<PPML_REAL>(PPML_REAL* rho, PPML_REAL* m, PPML_REAL* en, PPML_REAL* ei,
                                    BatchLo<PPML_REAL> lo, InstDev* inst, const int2* items,
                                    double gamma, double cfl, int max_steps, int nlmax, int nmax,
                                    int nitems, size_t smem, int threads, cudaStream_t st) {
  switch (threads) {
    case 256:
      return launch_cluster_nt<256>(rho, m, en, ei, lo, inst, items, gamma, cfl, max_steps, nlmax,
                                    nmax, nitems, smem, st);
    case 512:
      return launch_cluster_nt<512>(rho, m, en, ei, lo, inst, items, gamma, cfl, max_steps, nlmax,
                                    nmax, nitems, smem, st);
    case 1024:
      return launch_cluster_nt<1024>(rho, m, en, ei, lo, inst, items, gamma, cfl, max_steps, nlmax,
                                     nmax, nitems, smem, st);
    default:
      return ppml_fail(PPML_E_INVAL, "batch CTA size %d is not 256, 512 or 1024", threads);
  }
}

template <>
int launch_batch<PPML_REAL>(PPML_REAL* rho, PPML_REAL* m, PPML_REAL* en, PPML_REAL* ei,
                            BatchLo<PPML_REAL> lo, InstDev* inst, const int* order, double gamma,
                            double cfl, int max_steps, int nmax, int ninst, size_t smem,
                            int threads, cudaStream_t st) {
  switch (threads) {
    case 256:
      return launch_batch_nt<256>(rho, m, en, ei, lo, inst, order, gamma, cfl, max_steps, nmax, ninst,
                                  smem, st);
    case 512:
      return launch_batch_nt<512>(rho, m, en, ei, lo, inst, order, gamma, cfl, max_steps, nmax, ninst,
                                  smem, st);
    case 1024:
      return launch_batch_nt<1024>(rho, m, en, ei, lo, inst, order, gamma, cfl, max_steps, nmax,
                                   ninst, smem, st);
    default:
      return ppml_fail(PPML_E_INVAL, "batch CTA size %d is not 256, 512 or 1024", threads);
  }
}

}  // namespace ppml
