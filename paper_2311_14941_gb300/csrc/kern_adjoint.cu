// kern_adjoint.cu -- the discrete-adjoint reverse pass, the per-parameter gradient reduction and the
// parameter shifts.
#include <cuda_runtime.h>

#include "../../include/chem.h"
#include "kernels.cuh"

namespace chemgb {

// ---- discrete adjoint: resident blocks pull cells (longest tapes first).  Shared memory: the forward cell
// layout; the workspaces (AdjLayout offsets) and contraction workspaces are in global memory.
template <int kWarps>
__global__ void __launch_bounds__(32 * kWarps, 8 / kWarps)
k_adjoint(MechView M, AdjLayout A, int N, const double* __restrict__ p, const double* __restrict__ rec_h,
          const double* __restrict__ rec_ck, const int* __restrict__ rec_n, int K, const double* __restrict__ gT,
          const double* __restrict__ gY, double* __restrict__ grad_cell, double* __restrict__ gT0,
          double* __restrict__ gY0, int* __restrict__ status, int* __restrict__ head, const int* __restrict__ perm,
          double* ctr_ws, double* warp_ws, IntOpts o) {
  extern __shared__ double smem[];
  const int lane = threadIdx.x % kWarp;
  const int gw = blockIdx.x, w = threadIdx.x / kWarp;   // one cell per block
  double* s = smem;
  double* ctr = ctr_ws + (size_t)gw * kWarps * A.ctr;
  double* ws = warp_ws + (size_t)gw * (A.total + A.second);
  const int m = M.m;
  double* LAM = ws + A.LAM;
  double* GA = ws + A.GA;
  double* GE = ws + A.GE;
  double* GA2 = ws + A.total + A.GA2;
  double* GE2 = ws + A.total + A.GE2;
  auto clear = [&]() {   // every warp its own sums; one warp both
    if (w == 0)
      for (int r = lane; r < M.R; r += kWarp) { GA[r] = 0.0; GE[r] = 0.0; }
    if (w == kWarps - 1)
      for (int r = lane; r < M.R; r += kWarp) { GA2[r] = 0.0; GE2[r] = 0.0; }
    __syncwarp();
  };
  while (true) {
    int c = 0;
    if (threadIdx.x == 0) c = atomicAdd(head, 1);
    c = __shfl_sync(0xffffffffu, c, 0);
    if (kWarps > 1) {
      __shared__ int pulled;
      __syncthreads();   // warp 0 has taken the other's sums of the cell before
      if (threadIdx.x == 0) pulled = c;
      __syncthreads();
      c = pulled;
    }
    if (c >= N) break;
    c = perm[c];   // costliest cells (longest tapes) first
    const int na = rec_n[c];
    for (int i = lane; w == 0 && i < m; i += kWarp) LAM[i] = (i == 0) ? gT[c] : gY[(size_t)(i - 1) * N + c];
    clear();
    bool ok = na >= 0;
    if (ok) ok = adjoint_cell<kWarps>(M, s, ws, A, ctr, p[c], na, rec_h, rec_ck, K, N, c, Grp1{lane}, o, w);
    if (!ok) {
      for (int i = lane; w == 0 && i < m; i += kWarp) LAM[i] = 0.0;
      clear();
    }
    if (kWarps > 1) {
      __syncthreads();
      if (w != 0) continue;
    }
    for (int r = lane; r < M.R; r += kWarp) {
      const int d = __ldg(M.rx_order + r);
      grad_cell[(size_t)d * N + c] = GA[r] + GA2[r];
      grad_cell[(size_t)(M.R + d) * N + c] = GE[r] + GE2[r];
    }
    if (gT0 && lane == 0) gT0[c] = LAM[0];
    if (gY0)
      for (int i = 1 + lane; i < m; i += kWarp) gY0[(size_t)(i - 1) * N + c] = LAM[i];
    if (status && lane == 0 && !ok && status[c] == CHEM_CELL_OK) status[c] = CHEM_CELL_NOTAPE;
    __syncwarp();
  }
}

const void* adjoint_kernel(int warps) { return warps == 1 ? (const void*)k_adjoint<1> : (const void*)k_adjoint<2>; }

cudaError_t launch_adjoint(int warps, int grid, size_t smem, cudaStream_t stream, const MechView& M, const AdjLayout& A,
                           int N, const double* p, const double* rec_h, const double* rec_ck, const int* rec_n, int K,
                           const double* gT, const double* gY, double* grad_cell, double* gT0, double* gY0, int* status,
                           int* head, const int* perm, double* ctr_ws, double* warp_ws, const IntOpts& o) {
  const auto k = warps == 1 ? k_adjoint<1> : k_adjoint<2>;
  k<<<grid, warps * kWarp, smem, stream>>>(M, A, N, p, rec_h, rec_ck, rec_n, K, gT, gY, grad_cell, gT0, gY0, status,
                                           head, perm, ctr_ws, warp_ws, o);
  return cudaSuccess;
}

// sums over cells in a fixed order (one warp per parameter): deterministic gradients
__global__ void k_grad_reduce(int N, int P, const double* __restrict__ grad_cell, double* __restrict__ out1,
                              double* __restrict__ out2, int half) {
  const int wg = (blockIdx.x * blockDim.x + threadIdx.x) / kWarp, lane = threadIdx.x % kWarp;
  if (wg >= P) return;
  double acc = 0.0;
  for (int c = lane; c < N; c += kWarp) acc += grad_cell[(size_t)wg * N + c];
  acc = warp_sum(acc);
  if (lane == 0) {
    if (wg < half) out1[wg] = acc;
    else out2[wg - half] = acc;
  }
}

// parameter shifts: ln A_r = ln A_r,0 + dlnA[d], Ea_r = Ea_r,0 + dEa[d] (d: description index of
// compiled reaction r); Troe low-pressure limits shift jointly
__global__ void k_set_params(MechView M, const double* __restrict__ rxd0, double* __restrict__ rxd,
                             const double* __restrict__ dlnA, const double* __restrict__ dEa) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= M.R) return;
  const int d = __ldg(M.rx_order + r);
  const double a = dlnA ? dlnA[d] : 0.0, e = dEa ? dEa[d] / kRu : 0.0;
  const double* src = rxd0 + r;
  double* dst = rxd + r;
  dst[0] = src[0] + a;
  dst[2 * (size_t)M.R] = src[2 * (size_t)M.R] + e;
  if (__ldg((const int*)(M.rxi + (size_t)r * RX_I)) == 2) {
    dst[3 * (size_t)M.R] = src[3 * (size_t)M.R] + a;
    dst[5 * (size_t)M.R] = src[5 * (size_t)M.R] + e;
  }
}

}  // namespace chemgb
