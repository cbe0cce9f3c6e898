// kernels.cuh -- the integration, rate, Jacobian and adjoint kernels, declared for the C ABI.
//
// The kernels are compiled in several translation units (one per lane group of the integration kernels,
// kern_fwd_*.cu, and kern_adjoint.cu) so that the library builds in parallel; capi.cu launches them
// through these declarations.
#pragma once
#include "adjoint.cuh"
#include "device.cuh"

namespace chemgb {

__global__ void k_rates(MechView M, CellLayout L, int N, const double* __restrict__ T, const double* __restrict__ p,
                        const double* __restrict__ Y, double* __restrict__ dTdt, double* __restrict__ dYdt,
                        double* __restrict__ wdot);

__global__ void k_jacobian(MechView M, CellLayout L, int N, const double* __restrict__ T, const double* __restrict__ p,
                           const double* __restrict__ Y, double* __restrict__ Sv, double* __restrict__ u,
                           double* __restrict__ v);

// The integration kernels are templates on the lane group (one warp, two warps or half a warp per cell);
// their instantiations keep internal linkage inside their translation unit, so the ABI reaches them
// through these host functions (group g: 0 one warp, 1 two warps, 2 half a warp per cell; kNumGroups + i the
// i-th kernel with helper warps).
//   plain form: one lane group per cell, cells in index order;
//   persistent form: resident lane groups pull `chunk` cells at a time from the sorted queue `perm`.
enum ForwardKernel { KF_PLAIN = 0, KF_PERSISTENT = 1 };
// Host-side handle of the kernel (for cudaFuncSetAttribute, cudaFuncGetAttributes and occupancy queries).
const void* forward_kernel(ForwardKernel kind, int g);
cudaError_t launch_integrate_plain(int g, dim3 grid, dim3 block, size_t smem, cudaStream_t stream, const MechView& M,
                            const CellLayout& L, int N, double* T, const double* p, double* Y, const double* dt,
                            double* h_io, int* nsub, int* status, int* nacc_out, const IntOpts& o,
                            const unsigned long long* stamp, unsigned long long budget_ns);
cudaError_t launch_integrate_persistent(int g, dim3 grid, dim3 block, size_t smem, cudaStream_t stream, const MechView& M,
                                 const CellLayout& L, int N, double* T, const double* p, double* Y,
                                 const double* dt, double* h_io, int* nsub, int* status, int* nacc_out,
                                 const int* perm, unsigned long long* head, int chunk, const IntOpts& o,
                                 const unsigned long long* stamp, unsigned long long budget_ns);

// Per-group pieces, one translation unit each.
template <class Gp, class MV>
const void* plain_kernel();
template <class Gp, class MV>
const void* persistent_kernel();
template <class Gp, class MV>
cudaError_t launch_plain_g(dim3 grid, dim3 block, size_t smem, cudaStream_t stream, const MechView& M, const CellLayout& L,
                    int N, double* T, const double* p, double* Y, const double* dt, double* h_io, int* nsub,
                    int* status, int* nacc_out, const IntOpts& o, const unsigned long long* stamp,
                    unsigned long long budget_ns);
template <class Gp, class MV>
cudaError_t launch_persistent_g(dim3 grid, dim3 block, size_t smem, cudaStream_t stream, const MechView& M,
                         const CellLayout& L, int N, double* T, const double* p, double* Y, const double* dt,
                         double* h_io, int* nsub, int* status, int* nacc_out, const int* perm,
                         unsigned long long* head, int chunk, const IntOpts& o, const unsigned long long* stamp,
                         unsigned long long budget_ns);

// Discrete adjoint: resident blocks of one or two warps pull one cell at a time, longest tapes first; shared memory
// holds the forward cell layout (with two warps, a second dual-number cell behind it), a block's workspace (A.total
// doubles, then A.second for the sums of the second half of the second-order terms) and contraction workspaces (A.ctr per warp) are in global memory.
const void* adjoint_kernel(int warps);
cudaError_t launch_adjoint(int warps, int grid, size_t smem, cudaStream_t stream, const MechView& M, const AdjLayout& A,
                           int N, const double* p, const double* rec_h, const double* rec_ck, const int* rec_n, int K,
                           const double* gT, const double* gY, double* grad_cell, double* gT0, double* gY0, int* status,
                           int* head, const int* perm, double* ctr_ws, double* warp_ws, const IntOpts& o);

__global__ void k_grad_reduce(int N, int P, const double* __restrict__ grad_cell, double* __restrict__ out1,
                              double* __restrict__ out2, int half);

__global__ void k_set_params(MechView M, const double* __restrict__ rxd0, double* __restrict__ rxd,
                             const double* __restrict__ dlnA, const double* __restrict__ dEa);

}  // namespace chemgb
