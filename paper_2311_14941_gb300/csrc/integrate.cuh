// integrate.cuh -- the integration kernels (one lane group per cell), device code only.
//
// Templates on the lane group Gp (one warp, two warps or half a warp per cell), the mechanism view MV and
// the cell layout LT.  The library instantiates them with the run-time MechView / CellLayout; the
// mechanism-specialised build compiles the same source at run time with views whose sizes are
// compile-time constants (derived types with the same data members).  Nothing here may need a C library
// header, so the run-time compiler can take it as it is.
#pragma once
#include "device.cuh"

namespace chemgb {

__device__ __forceinline__ IntOpts with_deadline(IntOpts o, const unsigned long long* stamp,
                                                 unsigned long long budget_ns) {
  if (budget_ns && stamp) o.deadline_ns = *stamp + budget_ns;
  return o;
}

// Load one cell's state into y (lanes over state components).
template <class Gp>
__device__ __forceinline__ void load_state(double* y, int m, int N, int c, const double* T, const double* Y,
                                           const Gp& g) {
  for (int i = g.lane; i < m; i += g.size) y[i] = (i == 0) ? T[c] : Y[(size_t)(i - 1) * N + c];
  g.sync();
}

// The lane group of this thread (Gp: one warp, two warps or half a warp per cell); s = the cell's memory.
template <class LT>
__device__ __forceinline__ void cell_slot(int gs, const LT& L, double* smem, int& cell_in_block, double*& s) {
  cell_in_block = threadIdx.x / gs;
  s = smem + (size_t)cell_in_block * L.total;
}
template <class LT>
__device__ __forceinline__ Grp1 make_group(const Grp1*, const LT& L, double* smem, int& cell_in_block, double*& s) {
  cell_slot(Grp1::size, L, smem, cell_in_block, s);
  return Grp1{(int)threadIdx.x - cell_in_block * Grp1::size};
}
template <class LT>
__device__ __forceinline__ Grp2 make_group(const Grp2*, const LT& L, double* smem, int& cell_in_block, double*& s) {
  cell_slot(Grp2::size, L, smem, cell_in_block, s);
  return Grp2{(int)threadIdx.x - cell_in_block * Grp2::size, 1 + cell_in_block, s + L.misc};
}
template <class LT>
__device__ __forceinline__ GrpH make_group(const GrpH*, const LT& L, double* smem, int& cell_in_block, double*& s) {
  cell_slot(GrpH::size, L, smem, cell_in_block, s);
  const int half = (threadIdx.x / GrpH::size) & 1;
  return GrpH{(int)threadIdx.x - cell_in_block * GrpH::size, half ? 0xffff0000u : 0x0000ffffu};
}
template <class Gp, class LT>
__device__ __forceinline__ Gp cell_group(const LT& L, double* smem, int& cell_in_block, double*& s) {
  return make_group(static_cast<const Gp*>(nullptr), L, smem, cell_in_block, s);
}

// Block-cooperative coalesced load of the block's consecutive cells: adjacent threads read adjacent
// cells of the same state row (structure of arrays), then each lane group owns its cell's copy.
template <class LT>
__device__ __forceinline__ void load_tile(double* smem, const LT& L, int m, int N, int c0, int wpb, const double* T,
                                          const double* Y) {
  const int total = wpb * m;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int row = idx / wpb, w = idx - row * wpb;
    const int c = c0 + w;
    if (c < N) smem[(size_t)w * L.total + L.y + row] = (row == 0) ? T[c] : Y[(size_t)(row - 1) * N + c];
  }
  __syncthreads();
}

// Write a cell that has ended back to global memory.
template <class Gs, class MV, class LT>
__device__ __forceinline__ void store_cell(const MV& M, double* s, const LT& L, int N, const Gs& g, const CellRun& r,
                                           double* T, double* Y, double* h_io, int* nsub, int* status, int* nacc_out) {
  const SPtr y = shared_ptr(s) + L.y;
  const int c = r.cell;
  for (int i = g.lane; i < M.m; i += g.size) {
    if (i == 0) T[c] = y[0];
    else Y[(size_t)(i - 1) * N + c] = y[i];
  }
  if (g.lane == 0) {
    h_io[c] = r.h;
    nsub[c] = r.ns;
    status[c] = r.status;
    if (nacc_out) nacc_out[c] = r.na;
  }
}

// A state for a group that has no cell but shares its warp with one that has: the attempts it takes along must not
// meet infinities and NaN, whose handling is slow.
template <class Gp, class LT>
__device__ __forceinline__ void idle_state(double* s, const LT& L, int m, const Gp& g) {
  for (int i = g.lane; i < m; i += g.size) s[L.y + i] = i == 0 ? 1000.0 : 1.0 / (m - 1);
}

// Whole lane groups and whole warps; with helpers, one cell's warps and its helpers.
template <class Gp, class MV>
__device__ __forceinline__ bool block_shape() {
  if (MV::kHelpers > 0) return blockDim.x == Gp::size + MV::kHelpers * kWarp;
  return blockDim.x % Gp::size == 0 && blockDim.x % kWarp == 0;
}

// Plain form: one lane group per cell, cells in index order, one launch.
template <class Gp, class MV = MechView, class LT = CellLayout>
__global__ void k_integrate_plain(MV M, LT L, int N, double* __restrict__ T, const double* __restrict__ p,
                                  double* __restrict__ Y, const double* __restrict__ dt, double* __restrict__ h_io,
                                  int* __restrict__ nsub, int* __restrict__ status, int* __restrict__ nacc_out,
                                  IntOpts o, const unsigned long long* stamp, unsigned long long budget_ns) {
  extern __shared__ double smem[];
  if (!block_shape<Gp, MV>()) return;   // the launchers reject such shapes
  const int cpb = MV::kHelpers > 0 ? 1 : blockDim.x / Gp::size;
  int w = 0;
  double* s = nullptr;
  const Gp g = cell_group<Gp>(L, smem, w, s);
  const int c0 = blockIdx.x * cpb;
  load_tile(smem, L, M.m, N, c0, cpb, T, Y);
  if constexpr (MV::kHelpers > 0)
    if (threadIdx.x >= Gp::size) return help<Gp>(M, smem, L);
  const int c = c0 + w;
  const IntOpts oo = with_deadline(o, stamp, budget_ns);
  CellRun r;
  if (c < N) cell_start(M, s, L, c, p[c], dt[c], h_io[c], oo, solo(g), r);
  else idle_state(s, L, M.m, g);
  g.sync();
  while (any_cell(g, r.active)) cell_step(M, s, L, oo, g, r);
  if constexpr (MV::kHelpers > 0) help_end<Gp, MV::kHelpers>();
  if (c < N) {
    cell_end(oo, g, r);
    store_cell(M, s, L, N, g, r, T, Y, h_io, nsub, status, nacc_out);
  }
}

// Persistent form: grid sized to the resident capacity; every lane group pulls `chunk` cells at a time from the
// sorted queue with one atomicAdd and integrates them one after the other.  No block-wide barrier: warps of a
// block finish independently; groups that share a warp take their attempts together and pull whenever they have
// ended a cell.
template <class Gs>
__device__ __forceinline__ long long queue_pull(const Gs& g, unsigned long long* head, int chunk) {
  return gbcast(g, g.lane == 0 ? (long long)atomicAdd(head, (unsigned long long)chunk) : 0ll);
}

template <class Gp, class MV = MechView, class LT = CellLayout>
__global__ void k_integrate_persistent(MV M, LT L, int N, double* __restrict__ T, const double* __restrict__ p,
                                       double* __restrict__ Y, const double* __restrict__ dt,
                                       double* __restrict__ h_io, int* __restrict__ nsub, int* __restrict__ status,
                                       int* __restrict__ nacc_out, const int* __restrict__ perm,
                                       unsigned long long* __restrict__ head, int chunk, IntOpts o,
                                       const unsigned long long* stamp, unsigned long long budget_ns) {
  extern __shared__ double smem[];
  if (!block_shape<Gp, MV>()) return;   // the launchers reject such shapes
  if constexpr (MV::kHelpers > 0)
    if (threadIdx.x >= Gp::size) return help<Gp>(M, smem, L);
  int w = 0;
  double* s = nullptr;
  const Gp g = cell_group<Gp>(L, smem, w, s);
  const IntOpts oo = with_deadline(o, stamp, budget_ns);
  if (Gp::size < kWarp) idle_state(s, L, M.m, g);
  CellRun r;
  // 64-bit queue head: every pull adds `chunk`, including the last pulls past the end, so a 32-bit head could
  // wrap for large N * lane groups * chunk
  long long next = 0, end = 0;
  bool more = true;
  while (true) {
    const auto gs = solo(g);
    while (!r.active && more) {   // the next cell that has something to integrate
      if (next >= end) {
        next = queue_pull(gs, head, chunk);
        end = min(next + (long long)chunk, (long long)N);
        if (next >= N) { more = false; break; }
      }
      const int c = perm[next++];
      load_state(s + L.y, M.m, N, c, T, Y, gs);
      cell_start(M, s, L, c, p[c], dt[c], h_io[c], oo, gs, r);
      if (!r.active) {
        cell_end(oo, gs, r);
        store_cell(M, s, L, N, gs, r, T, Y, h_io, nsub, status, nacc_out);
        gs.sync();
      }
    }
    g.sync();
    if (!any_cell(g, r.active)) break;
    const bool was = r.active;
    cell_step(M, s, L, oo, g, r);
    if (was && !r.active) {
      cell_end(oo, gs, r);
      store_cell(M, s, L, N, gs, r, T, Y, h_io, nsub, status, nacc_out);
      gs.sync();
    }
  }
  if constexpr (MV::kHelpers > 0) help_end<Gp, MV::kHelpers>();
}

}  // namespace chemgb
