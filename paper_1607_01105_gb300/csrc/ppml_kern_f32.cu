// FP32 instantiation of the stencil kernels (FMA contraction on).
#include "ppml_tile_f32.cuh"

namespace ppml {
namespace {

cudaError_t prepare_sweeps(float) {
  cudaError_t e = cudaFuncSetAttribute(lagrangian_sweep_f32<false>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(SweepSmem));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(lagrangian_sweep_f32<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(SweepSmem));
  auto euler = [&](auto kernel) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)sizeof(EulerSmem));
  };
  euler(eulerian_sweep_f32<false, false>);
  euler(eulerian_sweep_f32<false, true>);
  euler(eulerian_sweep_f32<true, false>);
  euler(eulerian_sweep_f32<true, true>);
  return e;
}

// Three active axes, and offsets (three halo planes beyond the grid included) of 32 bits.
bool sweep_grid(const MarchArgs<float>& A) {
  return A.g.n[0] > 1 && A.g.n[1] > 1 && A.g.n[2] > 1 && offsets_fit(A.g);
}

// Eulerian stage of plain float states with three active axes.  False: not such a state.
bool launch_euler_sweeps(const MarchArgs<float>& A, int nblk, cudaStream_t st) {
  if (!sweep_grid(A)) return false;
  constexpr size_t SM = sizeof(EulerSmem);
  const bool flat = (A.flags & PPML_FIRST_ORDER) != 0;
  if (A.phi) {
    if (flat)
      eulerian_sweep_f32<true, true><<<nblk, TN, SM, st>>>(A);
    else
      eulerian_sweep_f32<false, true><<<nblk, TN, SM, st>>>(A);
  } else {
    if (flat)
      eulerian_sweep_f32<true, false><<<nblk, TN, SM, st>>>(A);
    else
      eulerian_sweep_f32<false, false><<<nblk, TN, SM, st>>>(A);
  }
  return true;
}

// Lagrangian stage of plain float states with three active axes: face velocities, then the
// sweeps; in several launches of about as many tiles each where the face array does not hold
// every tile (the allocation-free step, or a grid whose tiles are mostly padding), then in
// x-major order (the results do not depend on it).  False: not such a state, nothing launched.
bool launch_sweeps(const MarchArgs<float>& A, int nblk, cudaStream_t st) {
  if (!A.face || !sweep_grid(A)) return false;
  MarchArgs<float> B = A;
  const int tiles = A.tiles_x * A.tiles_y * A.tiles_z;
  int per = nblk;  // (padded orders launch more blocks than there are tiles)
  if (A.face_tiles < tiles) {
    B.tile_order = 0;
    nblk = tiles;
    const int launches = (tiles + A.face_tiles - 1) / A.face_tiles;
    per = (tiles + launches - 1) / launches;
  }
  for (int first = 0; first < nblk; first += per) {
    const int n = nblk - first < per ? nblk - first : per;
    B.tile_first = first;
    B.face_first = first;
    face_velocity_f32<<<n, FV_THREADS, 0, st>>>(B);
    if (A.flags & PPML_FIRST_ORDER)
      lagrangian_sweep_f32<true><<<n, TN, sizeof(SweepSmem), st>>>(B);
    else
      lagrangian_sweep_f32<false><<<n, TN, sizeof(SweepSmem), st>>>(B);
  }
  return true;
}

}  // namespace
}  // namespace ppml

#define PPML_REAL float
#include "ppml_kern_impl.cuh"
