// kern_forward.cuh -- host-side handles and launchers of the integration kernels (integrate.cuh), included
// by one translation unit per lane group and form (kern_fwd_warp*.cu, kern_fwd_pair.cu, kern_fwd_half.cu).
#pragma once
#include <cuda_runtime.h>

#include "../../include/chem.h"
#include "integrate.cuh"
#include "kernels.cuh"

namespace chemgb {

template <class Gp, class MV>
bool launch_shape(dim3 block) {
  if (block.y != 1 || block.z != 1) return false;
  if (MV::kHelpers > 0) return block.x == Gp::size + MV::kHelpers * kWarp;
  return block.x % Gp::size == 0 && block.x % kWarp == 0;
}

// Host-side handles and launches of the instantiations for lane group Gp (explicitly instantiated in one
// translation unit per group and form).
template <class Gp, class MV>
const void* plain_kernel() {
  return (const void*)k_integrate_plain<Gp, MV>;
}

template <class Gp, class MV>
const void* persistent_kernel() {
  return (const void*)k_integrate_persistent<Gp, MV>;
}

template <class Gp, class MV>
cudaError_t launch_plain_g(dim3 grid, dim3 block, size_t smem, cudaStream_t stream, const MechView& M,
                           const CellLayout& L, int N, double* T, const double* p, double* Y, const double* dt,
                           double* h_io, int* nsub, int* status, int* nacc_out, const IntOpts& o,
                           const unsigned long long* stamp, unsigned long long budget_ns) {
  if (!launch_shape<Gp, MV>(block)) return cudaErrorInvalidValue;
  MV v;
  static_cast<MechView&>(v) = M;
  k_integrate_plain<Gp, MV><<<grid, block, smem, stream>>>(v, L, N, T, p, Y, dt, h_io, nsub, status, nacc_out, o, stamp,
                                                       budget_ns);
  return cudaSuccess;
}

template <class Gp, class MV>
cudaError_t launch_persistent_g(dim3 grid, dim3 block, size_t smem, cudaStream_t stream, const MechView& M,
                                const CellLayout& L, int N, double* T, const double* p, double* Y, const double* dt,
                                double* h_io, int* nsub, int* status, int* nacc_out, const int* perm,
                                unsigned long long* head, int chunk, const IntOpts& o,
                                const unsigned long long* stamp, unsigned long long budget_ns) {
  if (!launch_shape<Gp, MV>(block)) return cudaErrorInvalidValue;
  MV v;
  static_cast<MechView&>(v) = M;
  k_integrate_persistent<Gp, MV><<<grid, block, smem, stream>>>(v, L, N, T, p, Y, dt, h_io, nsub, status, nacc_out, perm,
                                                            head, chunk, o, stamp, budget_ns);
  return cudaSuccess;
}

}  // namespace chemgb
