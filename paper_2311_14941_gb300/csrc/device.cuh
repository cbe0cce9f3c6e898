// device.cuh -- warp-level device routines: one warp owns one reactor cell, its state and its sparse
// factor in shared memory.
//
// Mathematical content (the paper names the techniques, Sec. 2.5; the formulas are the standard ones):
//   f(y):  y = (T, Y_1..Y_n) at fixed p.  C_k = rho Y_k / W_k, rho = p Wbar / (Ru T).
//          k_f = exp(ln A + b ln T - Ea/(Ru T)); third-body [M]; Troe fall-off; k_r = k_f / Kc with
//          1/Kc = prod_k exp(g_k)^nu_k (Ru T / p0)^(sum nu), g_k = h_k/(Ru T) - s_k/Ru (NASA-7), so a
//          reaction's reverse rate costs multiplications only (one exp per species, not per reaction).
//          dY_k/dt = W_k w_k / rho,  dT/dt = -sum_k H_k w_k / (rho c_p).
//   J(y):  exact Jacobian written as S + u v^T.  With [M] = p/(Ru T) + sum_listed (alpha_j - 1) C_j (the
//          default efficiencies add up to the total concentration, a function of T alone at fixed p),
//          d w / d C is sparse: Dtil = sum_r nu_r (d q_r / d C).  Then, with g_k = sum_j Dtil_kj C_j,
//            S_kj = (W_k/W_j) Dtil_kj,  u_k = (W_k/rho)(w_k - g_k),  v_j = Wbar / W_j,
//            S_kT = (W_k/rho)(w_T,k - g_k/T) + f_k/T      (w_T = d w / d T at fixed C)
//            S_Tj = -(Ru T sum_k hRT_k Dtil_kj + f_T cpR_j Ru) / (W_j c_p)
//            S_TT = -sum_k [Cp_k w_k + H_k (w_T,k - g_k/T)] / (rho c_p) + f_T (1/T - Ru sum Y dcpR/dT / W / c_p)
//            u_T  = sum_k H_k g_k / (rho c_p) + f_T.
//   Step:  RODAS3 (Sandu et al. 1997) in the transformed form of Hairer & Wanner (Vol. II, IV.7):
//            (I/(h gamma) - J) U_i = f(y + sum_j a_ij U_j) + sum_j (c_ij / h) U_j,
//            y_new = y + sum m_i U_i,  err = sum e_i U_i,
//          where J = S + u v^T is inverted by Sherman-Morrison around the sparse LU of I/(h gamma) - S.
#pragma once
#include "mech.h"
#include "scalar.cuh"

namespace chemgb {

// -------------------------------------------------------------------------------------- lane groups
// The lanes that integrate one cell: one warp (GrpW<1>), or two consecutive warps of a block (GrpW<2>).
// Work inside a cell is strided over the group's lanes; shared-memory ordering inside the group is a
// warp barrier for one warp and a named barrier (bar.sync id, 64) for two.  Reductions add each warp's
// butterfly sum in warp order, so every lane of the group holds the same, reproducible value.  The
// group size is a compile-time constant: the one-warp code is the plain warp code.
template <int W>
struct GrpW;

template <>
struct GrpW<1> {
  static constexpr int size = kWarp;
  int lane;
  __device__ __forceinline__ void sync() const { __syncwarp(); }
};

template <>
struct GrpW<2> {
  static constexpr int size = 2 * kWarp;
  int lane;     // 0 .. 63
  int bar;      // named barrier of the group: 1 + the cell's index in its block
  double* xch;  // one exchange slot per warp in the cell's shared memory
  __device__ __forceinline__ void sync() const {
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(size) : "memory");
  }
};

using Grp1 = GrpW<1>;
using Grp2 = GrpW<2>;

// Half a warp: two cells share a warp, 16 lanes each (mechanisms with few species, whose loops and sparse programs
// leave most of a warp's lanes idle).  The two cells take every attempt together (see cell_step): an FP64
// instruction takes the pipe for 64 cycles however many lanes it has, so run apart they would pay for each other
// (6,000 cells of 10 species / 27 reactions: 368 ms apart, 346 together).
// GrpH is such a half inside an attempt: the whole warp takes part in every barrier and vote.  GrpHs is the half by
// itself (starting and finishing its cell).
struct GrpHs {
  static constexpr int size = kWarp / 2;
  int lane;        // 0 .. 15
  unsigned mask;   // the lanes of this half of the warp
  __device__ __forceinline__ void sync() const { __syncwarp(mask); }
};
struct GrpH {
  static constexpr int size = kWarp / 2;
  int lane;        // 0 .. 15
  unsigned mask;   // the lanes of this half of the warp
  __device__ __forceinline__ void sync() const { __syncwarp(); }
};
__device__ __forceinline__ const Grp1& solo(const Grp1& g) { return g; }
__device__ __forceinline__ const Grp2& solo(const Grp2& g) { return g; }
__device__ __forceinline__ GrpHs solo(const GrpH& g) { return GrpHs{g.lane, g.mask}; }
// Whether ok holds for one, for all of the cells of this warp (every lane of a cell passes the same value).
__device__ __forceinline__ bool any_cell(const Grp1&, bool ok) { return ok; }
__device__ __forceinline__ bool any_cell(const Grp2&, bool ok) { return ok; }
__device__ __forceinline__ bool any_cell(const GrpH&, bool ok) { return __any_sync(0xffffffffu, ok); }
__device__ __forceinline__ bool all_cells(const Grp1&, bool ok) { return ok; }
__device__ __forceinline__ bool all_cells(const Grp2&, bool ok) { return ok; }
__device__ __forceinline__ bool all_cells(const GrpH&, bool ok) { return __all_sync(0xffffffffu, ok); }

// Ordering among the lanes of half a group (both halves run the same steps, so a barrier of the whole warp will do;
// the halves of two warps are the warps themselves).
struct SyncMask {
  unsigned mask;
  __device__ __forceinline__ void sync() const { __syncwarp(mask); }
};
__device__ __forceinline__ SyncMask half_sync(const Grp1&) { return SyncMask{0xffffffffu}; }
__device__ __forceinline__ SyncMask half_sync(const Grp2&) { return SyncMask{0xffffffffu}; }
__device__ __forceinline__ SyncMask half_sync(const GrpH&) { return SyncMask{0xffffffffu}; }

__device__ __forceinline__ double gsum(const Grp1&, double v) { return warp_sum(v); }
__device__ __forceinline__ double gsum(const GrpH&, double v) {   // exchanges stay within the half
#pragma unroll
  for (int o = GrpH::size / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double gsum(const GrpHs& g, double v) {
#pragma unroll
  for (int o = GrpHs::size / 2; o > 0; o >>= 1) v += __shfl_xor_sync(g.mask, v, o);
  return v;
}
__device__ __forceinline__ double gsum(const Grp2& g, double v) {
  v = warp_sum(v);
  g.sync();   // earlier readers of the slots are done
  if ((g.lane & (kWarp - 1)) == 0) g.xch[g.lane / kWarp] = v;
  g.sync();
  return g.xch[0] + g.xch[1];
}
template <class G>
__device__ __forceinline__ Dual gsum(const G& g, Dual v) { return Dual(gsum(g, v.v), gsum(g, v.d)); }
template <class G, int K>
__device__ __forceinline__ DualN<K> gsum(const G& g, DualN<K> v) {
  v.v = gsum(g, v.v);
#pragma unroll
  for (int i = 0; i < K; ++i) v.d[i] = gsum(g, v.d[i]);
  return v;
}

// Two or three sums in one butterfly.  After the first exchange the lower half of the lanes carries the first
// value and the upper half the second, so the remaining exchanges add both at once (and the third value joins
// them after its second exchange): 5 additions on the FP64 pipe for two warp-wide sums instead of 10, 7 for three
// instead of 15.  Every lane adds the same pairs in the same order as the single sums, so the results are theirs.
template <int W>
__device__ __forceinline__ void bfly2(unsigned mask, int lane, double& a, double& b) {
  const bool up = (lane & (W / 2)) != 0;
  double v = (up ? b : a) + __shfl_xor_sync(mask, up ? a : b, W / 2);
#pragma unroll
  for (int o = W / 4; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
  a = __shfl_sync(mask, v, 0, W);
  b = __shfl_sync(mask, v, W / 2, W);
}
template <int W>
__device__ __forceinline__ void bfly3(unsigned mask, int lane, double& a, double& b, double& c) {
  const bool up = (lane & (W / 2)) != 0, up2 = (lane & (W / 4)) != 0;
  double v = (up ? b : a) + __shfl_xor_sync(mask, up ? a : b, W / 2);
  c += __shfl_xor_sync(mask, c, W / 2);
  v = (up2 ? c : v) + __shfl_xor_sync(mask, up2 ? v : c, W / 4);
#pragma unroll
  for (int o = W / 8; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
  a = __shfl_sync(mask, v, 0, W);
  b = __shfl_sync(mask, v, W / 2, W);
  c = __shfl_sync(mask, v, W / 4, W);
}
__device__ __forceinline__ void gsum2(const Grp1& g, double& a, double& b) { bfly2<kWarp>(0xffffffffu, g.lane, a, b); }
__device__ __forceinline__ void gsum2(const GrpH& g, double& a, double& b) { bfly2<GrpH::size>(0xffffffffu, g.lane, a, b); }
__device__ __forceinline__ void gsum3(const Grp1& g, double& a, double& b, double& c) {
  bfly3<kWarp>(0xffffffffu, g.lane, a, b, c);
}
__device__ __forceinline__ void gsum3(const GrpH& g, double& a, double& b, double& c) {
  bfly3<GrpH::size>(0xffffffffu, g.lane, a, b, c);
}
__device__ __forceinline__ void gsum2(const Grp2& g, double& a, double& b) {
  bfly2<kWarp>(0xffffffffu, g.lane & (kWarp - 1), a, b);
  g.sync();   // earlier readers of the slots are done
  if ((g.lane & (kWarp - 1)) == 0) { g.xch[g.lane / kWarp] = a; g.xch[2 + g.lane / kWarp] = b; }
  g.sync();
  a = g.xch[0] + g.xch[1];
  b = g.xch[2] + g.xch[3];
}
__device__ __forceinline__ void gsum3(const Grp2& g, double& a, double& b, double& c) {
  bfly3<kWarp>(0xffffffffu, g.lane & (kWarp - 1), a, b, c);
  g.sync();   // earlier readers of the slots are done
  if ((g.lane & (kWarp - 1)) == 0) {
    g.xch[g.lane / kWarp] = a; g.xch[2 + g.lane / kWarp] = b; g.xch[4 + g.lane / kWarp] = c;
  }
  g.sync();
  a = g.xch[0] + g.xch[1];
  b = g.xch[2] + g.xch[3];
  c = g.xch[4] + g.xch[5];
}
template <class G, class Sc>   // dual numbers: one sum after the other
__device__ __forceinline__ void gsum2(const G& g, Sc& a, Sc& b) { a = gsum(g, a); b = gsum(g, b); }
template <class G, class Sc>
__device__ __forceinline__ void gsum3(const G& g, Sc& a, Sc& b, Sc& c) { a = gsum(g, a); b = gsum(g, b); c = gsum(g, c); }

__device__ __forceinline__ bool gall(const Grp1&, bool ok) { return __all_sync(0xffffffffu, ok); }
__device__ __forceinline__ bool gall(const GrpHs& g, bool ok) { return __all_sync(g.mask, ok); }
__device__ __forceinline__ bool gall(const GrpH& g, bool ok) { return (__ballot_sync(0xffffffffu, ok) & g.mask) == g.mask; }
__device__ __forceinline__ bool gall(const Grp2& g, bool ok) {
  ok = __all_sync(0xffffffffu, ok);
  g.sync();
  if ((g.lane & (kWarp - 1)) == 0) g.xch[g.lane / kWarp] = ok ? 1.0 : 0.0;
  g.sync();
  return g.xch[0] != 0.0 && g.xch[1] != 0.0;
}

// Whether ok holds on all lanes of the group that share this thread's warp (all of them call it).
__device__ __forceinline__ bool wall(const Grp1&, bool ok) { return __all_sync(0xffffffffu, ok); }
__device__ __forceinline__ bool wall(const GrpH&, bool ok) { return __all_sync(0xffffffffu, ok); }
__device__ __forceinline__ bool wall(const Grp2&, bool ok) { return __all_sync(0xffffffffu, ok); }

// The value of lane 0, on every lane of the group.
__device__ __forceinline__ long long gbcast(const Grp1&, long long v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ long long gbcast(const GrpHs& g, long long v) { return __shfl_sync(g.mask, v, 0, GrpHs::size); }
__device__ __forceinline__ long long gbcast(const Grp2& g, long long v) {
  g.sync();
  if (g.lane == 0) g.xch[0] = __longlong_as_double(v);
  g.sync();
  const long long r = __double_as_longlong(g.xch[0]);
  g.sync();   // everyone has read the slot before it is reused
  return r;
}

// RODAS3 in transformed form.  a = alpha Gamma^-1, c = diag(1/gamma) - Gamma^-1, m = b Gamma^-1,
// e = (b - bhat) Gamma^-1, obtained from the published alpha_ij, gamma_ij, b, bhat (gamma = 1/2).
// Zero coefficients are exploited below: a21 = a32 = a42 = 0 (stage 2 reuses f(y)), m2 = 0,
// e = (0, 0, 0, 1).
constexpr double RG = 0.5;
constexpr double A31 = 2.0, A41 = 2.0, A43 = 1.0;
constexpr double C21 = 4.0, C31 = 1.0, C32 = -1.0, C41 = 1.0, C42 = -1.0, C43 = -8.0 / 3.0;
constexpr double M1 = 2.0, M3 = 1.0, M4 = 1.0;

// ROS2 (Verwer, Spee, Blom and Hundsdorfer 1999), order 2 with a first-order embedded solution,
// L-stable with gamma = 1 + 1/sqrt(2).  Its published stages (I - gamma h J) k1 = f(y),
// (I - gamma h J) k2 = f(y + h k1) - 2 k1 give, with U_i = gamma h k_i, the transformed form
//   (I/(h gamma) - J) U1 = f(y),  (I/(h gamma) - J) U2 = f(y + U1/gamma) - (2/(gamma h)) U1,
//   y_new = y + (3/(2 gamma)) U1 + (1/(2 gamma)) U2,  err = (U1 + U2)/(2 gamma).
constexpr double RG2 = 0x1.b504f333f9de6p+0;   // 1 + 1/sqrt(2) rounded to double
constexpr double R2_A21 = 1.0 / RG2, R2_C21 = -2.0 / RG2, R2_M1 = 1.5 / RG2, R2_M2 = 0.5 / RG2, R2_E = 0.5 / RG2;

// RODAS4 (Hairer and Wanner, Solving ODEs II, Sec. VI.4), order 4 with an order-3 embedded solution,
// stiffly accurate and L-stable, gamma = 1/4, in its published transformed form:
//   (I/(h gamma) - J) U_i = f(y + sum_j a_ij U_j) + sum_j (c_ij / h) U_j.
// a_6j = a_5j (j < 5) and a_65 = 1, m = (a_51, a_52, a_53, a_54, 1, 1), e = (0, 0, 0, 0, 0, 1): stage 6
// starts from stage 5's point plus U5, y_new is stage 6's point plus U6, and U6 is the error estimate.
constexpr double RG4 = 0.25;
constexpr double R4_A21 = 1.544;
constexpr double R4_A31 = 0.9466785280815826, R4_A32 = 0.2557011698983284;
constexpr double R4_A41 = 3.314825187068521, R4_A42 = 2.896124015972201, R4_A43 = 0.9986419139977817;
constexpr double R4_A51 = 1.221224509226641, R4_A52 = 6.019134481288629, R4_A53 = 12.53708332932087,
                 R4_A54 = -0.6878860361058950;
constexpr double R4_C21 = -5.6688;
constexpr double R4_C31 = -2.430093356833875, R4_C32 = -0.2063599157091915;
constexpr double R4_C41 = -0.1073529058151375, R4_C42 = -9.594562251023355, R4_C43 = -20.47028614809616;
constexpr double R4_C51 = 7.496443313967647, R4_C52 = -10.24680431464352, R4_C53 = -33.99990352819905,
                 R4_C54 = 11.70890893206160;
constexpr double R4_C61 = 8.083246795921522, R4_C62 = -7.981132988064893, R4_C63 = -31.52159432874371,
                 R4_C64 = 16.31930543123136, R4_C65 = -6.058818238834054;
// The three methods as tables for one stage loop (constant memory, read with warp-uniform indices).  Row k - 2 of
// stage k: the point y + sum_j a_kj U_j in ascending j (zero coefficients are skipped) and the coefficient sum
// sum_j c_kj U_j in descending j.  RODAS3's stage 2 has no point of its own (a21 = 0: f(y) again).
static __constant__ double kR4A[4][4] = {{R4_A21, 0.0, 0.0, 0.0},
                                         {R4_A31, R4_A32, 0.0, 0.0},
                                         {R4_A41, R4_A42, R4_A43, 0.0},
                                         {R4_A51, R4_A52, R4_A53, R4_A54}};
static __constant__ double kR4C[5][5] = {{R4_C21, 0.0, 0.0, 0.0, 0.0},
                                         {R4_C31, R4_C32, 0.0, 0.0, 0.0},
                                         {R4_C41, R4_C42, R4_C43, 0.0, 0.0},
                                         {R4_C51, R4_C52, R4_C53, R4_C54, 0.0},
                                         {R4_C61, R4_C62, R4_C63, R4_C64, R4_C65}};
// methods 0 (RODAS3) and 1 (ROS2)
static __constant__ double kRosA[2][3][3] = {{{0.0, 0.0, 0.0}, {A31, 0.0, 0.0}, {A41, 0.0, A43}},
                                             {{R2_A21, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}}};
static __constant__ double kRosC[2][3][3] = {{{C21, 0.0, 0.0}, {C31, C32, 0.0}, {C41, C42, C43}},
                                             {{R2_C21, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}}};
__device__ __forceinline__ double stage_a(int method, int k, int j) {   // a of stage k + 1 and U_(j+1)
  return method == 2 ? kR4A[k - 1][j] : kRosA[method][k - 1][j];
}
__device__ __forceinline__ double stage_c(int method, int k, int j) {
  return method == 2 ? kR4C[k - 1][j] : kRosC[method][k - 1][j];
}

constexpr double kInvLn10 = 0.43429448190325182765;
constexpr double kLn10 = 2.30258509299404568402;


// ---- doubles in shared memory by 32-bit address.  The compiler carries a pointer into shared memory as a 64-bit
// number and rebuilds addresses in 64 bits; a step of a substitution takes 166 cycles with plain pointers and 130
// with these.  The accesses are volatile and name memory as clobbered: they keep their order among themselves, around
// barriers and against plain accesses of the same cell, which they do not show the compiler otherwise (the clobber costs
// neither registers nor time).  The rate code, with many independent loads in flight, would pay for that order: it keeps
// plain pointers.  Between lanes, a barrier stands between one kind of access and the other, as between any two.
struct SRef {
  uint32_t a;
  __device__ __forceinline__ operator double() const {
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
  }
  __device__ __forceinline__ SRef& operator=(double v) {
    asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
    return *this;
  }
  __device__ __forceinline__ SRef& operator=(const SRef& o) { return *this = (double)o; }
  __device__ __forceinline__ SRef& operator+=(double v) { return *this = (double)*this + v; }
  __device__ __forceinline__ SRef& operator*=(double v) { return *this = (double)*this * v; }
};
struct SPtr {
  uint32_t a;
  __device__ __forceinline__ SRef operator[](int i) const { return SRef{a + (uint32_t)i * 8u}; }
  __device__ __forceinline__ SPtr operator+(int i) const { return SPtr{a + (uint32_t)i * 8u}; }
  __device__ __forceinline__ SPtr operator-(int i) const { return SPtr{a - (uint32_t)i * 8u}; }
};
__device__ __forceinline__ SPtr shared_ptr(const double* p) { return SPtr{(uint32_t)__cvta_generic_to_shared(p)}; }
// A cell's memory as the programs address it: shared memory for doubles, global memory for dual numbers.
__device__ __forceinline__ SPtr prog_ptr(double* p) { return shared_ptr(p); }
template <class T>
__device__ __forceinline__ T* prog_ptr(T* p) { return p; }
// Stores under a predicate, as one predicated instruction (the compiler makes a branch of an if, at about 60 cycles
// when lanes disagree).
__device__ __forceinline__ void store_if(const SPtr& p, int i, double v, bool yes) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %2, 0;\n\t@q st.shared.f64 [%0], %1;\n\t}" ::"r"(p.a + (uint32_t)i * 8u),
               "d"(v), "r"((int)yes) : "memory");
}
template <class T>
__device__ __forceinline__ void store_if(T* p, int i, const T& v, bool yes) {
  if (yes) p[i] = v;
}
// The number type behind a pointer (the routines below take plain pointers too: dual numbers and the adjoint's
// records live in global memory).
template <class P>
struct pointee;
template <>
struct pointee<SPtr> {
  using type = double;
};
template <class T>
struct pointee<T*> {
  using type = T;
};
template <class T>
struct pointee<const T*> {
  using type = T;
};
template <class P>
using num = typename pointee<P>::type;


// ---- running the warp programs.  A program is tens of kilobytes, more than the L1 that the cells' shared memory
// leaves, so every step's ops come from L2, 300 to 600 cycles away.  The steps are therefore taken in blocks of
// kProgBlock: a lane loads its ops of the next block (independent loads) before it executes the current one.  A
// step has no branch (a divergent branch costs about 60 cycles, as much as its FP64 instruction): idle lanes take
// part and do not store.  A step of the elimination so takes 125 to 155 cycles, of which 64 are the FP64
// instruction; read two steps ahead in a loop over kinds it took 640 in the kernel (one warp on an SM), ops included.
__device__ __forceinline__ GatherOp as_gop(uint2 v) {
  GatherOp o;
  o.a = (uint16_t)(v.x & 0xFFFF); o.b = (uint16_t)(v.x >> 16);
  o.dst = (uint16_t)(v.y & 0xFFFF); o.flags = (uint16_t)(v.y >> 16);
  return o;
}

// v <- the program's result.  A: the factor; lane of width: this lane's place among the program's lanes.  RECIP:
// elimination (v = A), false if a reciprocal is not finite.
template <bool RECIP, class Sy>
__device__ __forceinline__ bool run_fma(const FmaProgram& P, SPtr A, SPtr v, int lane, int width, const Sy& sy) {
  constexpr int slots = kProgBlock + (RECIP ? 1 : 0);
  bool ok = true;
  if (P.blocks <= 0) return ok;
  const uint2* op = reinterpret_cast<const uint2*>(P.ops) + lane;
  uint2 cur[slots], nxt[slots];
#pragma unroll
  for (int u = 0; u < slots; ++u) nxt[u] = __ldg(op + u * width);
  int head = RECIP ? __ldg(P.head) : 0;
  auto step = [&](uint2 w) {
    const int t = w.x & 0xFFFF, a = w.x >> 16, b = w.y & 0xFFFF;
    const double old = v[t], c = A[a], x = v[b];
    const double r = fma(-c, x, (w.y & (FM_MUL << 16)) ? -0.0 : old);
    if (!(w.y & (FM_IDLE << 16))) v[t] = r;
    sy.sync();
  };
#pragma unroll 1
  for (int blk = 0; blk < P.blocks; ++blk) {
    const int h = head;
#pragma unroll
    for (int u = 0; u < slots; ++u) cur[u] = nxt[u];
    if (blk + 1 < P.blocks) {
      op += slots * width;
      if (RECIP) head = __ldg(P.head + blk + 1);
#pragma unroll
      for (int u = 0; u < slots; ++u) nxt[u] = __ldg(op + u * width);
    }
    if (!RECIP) {   // whole blocks (the first slots of the last one may be idle)
#pragma unroll
      for (int u = 0; u < kProgBlock; ++u) step(cur[u]);
    } else {
      switch (h & 255) {
        case 8: step(cur[0]);   // fall through: the last h & 255 slots
        case 7: step(cur[1]);
        case 6: step(cur[2]);
        case 5: step(cur[3]);
        case 4: step(cur[4]);
        case 3: step(cur[5]);
        case 2: step(cur[6]);
        case 1: step(cur[7]);
        default: break;
      }
    }
    if (RECIP && (h & 256)) {
      const uint2 w = cur[slots - 1];
      const double r = rcp_rn(v[w.x >> 16]);
      if (!(w.y & (FM_IDLE << 16))) {
        ok = ok && finite_bits(r);   // 1/0 is infinite
        v[w.x & 0xFFFF] = -r;
      }
      sy.sync();
    }
  }
  return ok;
}

// Per-cell scalars shared by all lanes (every lane holds the same values).  tj, ttau: interval and local
// coordinate of T in the tables of tabulated temperature functions (tj < 0: exact evaluation).
template <class Sc>
struct ScalT {
  Sc T, lnT, invT, Wbar, rho, irho, cp, ctot, rtp, irtp, dcps;
  int tj;
  double ttau;
};

template <class A, class B>
struct same_type {
  static constexpr bool value = false;
};
template <class A>
struct same_type<A, A> {
  static constexpr bool value = true;
};
template <class Sc>
__host__ __device__ constexpr bool is_real() { return same_type<Sc, double>::value; }

// Polynomial in tau with coefficients c[0..d] (table memory, read-only path).
__device__ __forceinline__ double tab_poly(const double* c, int d, double tau) {
  double v = __ldg(c + d);
  for (int i = d - 1; i >= 0; --i) v = fma(v, tau, __ldg(c + i));
  return v;
}

// The table coordinates of T: interval j of u = 1/T and tau = 2 (u - u_j)/du - 1 (-1 outside the range or
// without tables; computed with the division, so that every implementation of the tables locates T alike).
template <class MV>
__device__ __forceinline__ void tab_locate(const MV& M, double T, double invT, int& tj, double& ttau) {
  tj = -1;
  ttau = 0.0;
  if (M.tab_on && T >= M.tab_tlo && T < M.tab_thi) {
    const double x = div_rn(invT - M.tab_ulo, M.tab_du);
    const int j = min(M.tab_ni - 1, max(0, (int)floor(x)));
    tj = j;
    ttau = 2.0 * (x - j) - 1.0;
  }
}
using Scal = ScalT<double>;

// Coefficient nu of the omega and Dtil gather programs: the op carries the top 16 bits of the IEEE
// double nu (exact for +-1, +-2, +-3), rebuilt with integer instructions (no conversion on the FP64 pipe).
__device__ __forceinline__ double nu_of(int b) { return __hiloint2double(b << 16, 0); }

// -------------------------------------------------------------------------------------- gathers
// out[g] = sum over the group's terms of val(a, b); partial sums of split groups are combined after.
// ADD: out[g] += sum instead (outputs without terms in the program are left as they are; its pieces end on common
// steps, marked in every lane's op).  ld(a, b) reads a term's operands, fin(operands, b) multiplies them.
//
// Doubles: a block of steps at a time.  The operands of the block are read before its sums, which are a chain of
// FP64 instructions with nothing to wait for.
template <bool ADD, class P, class PP, class Ld, class Fin, class Gp, class GT>
__device__ __forceinline__ void gather_blocks(const GT& G, P out, PP part, Ld ld, Fin fin, const Gp& g) {
  using Sc = num<P>;
  Sc acc = Sc(0.0);
  const uint2* op = reinterpret_cast<const uint2*>(G.ops) + g.lane;
  uint2 nxt[kProgBlock];
  if (G.blocks > 0) {
#pragma unroll
    for (int u = 0; u < kProgBlock; ++u) nxt[u] = __ldg(op + u * g.size);
  }
#pragma unroll 1
  for (int blk = 0; blk < G.blocks; ++blk) {
    uint2 cur[kProgBlock];
    decltype(ld(0, 0)) x[kProgBlock];
#pragma unroll
    for (int u = 0; u < kProgBlock; ++u) {
      cur[u] = nxt[u];
      x[u] = ld((int)(cur[u].x & 0xFFFF), (int)(cur[u].x >> 16));
    }
    if (blk + 1 < G.blocks) {
      op += kProgBlock * g.size;
#pragma unroll
      for (int u = 0; u < kProgBlock; ++u) nxt[u] = __ldg(op + u * g.size);
    }
#pragma unroll
    for (int u = 0; u < kProgBlock; ++u) {
      const GatherOp o = as_gop(cur[u]);
      const Sc sum = acc + fin(x[u], (int)o.b);
      if (!(o.flags & GF_IDLE)) acc = sum;
      const bool end = o.dst != DST_NONE, partial = (o.dst & PARTIAL_BIT) != 0;
      if (ADD) {
        if (o.flags & GF_END) {
          const Sc old = out[partial ? 0 : (int)o.dst];
          store_if(out, o.dst, old + acc, !partial);
          store_if(part, o.dst & 0x7FFF, acc, end && partial);
          if (end) acc = Sc(0.0);
        }
      } else {
        store_if(out, o.dst, acc, !partial);
        store_if(part, o.dst & 0x7FFF, acc, end && partial);
        if (end) acc = Sc(0.0);
      }
    }
  }
}
// Dual numbers: step by step (a step is long, and the operands of a block would spill).
template <bool ADD, class P, class PP, class Ld, class Fin, class Gp, class GT>
__device__ __forceinline__ void gather_steps(const GT& G, P out, PP part, Ld ld, Fin fin, const Gp& g) {
  using Sc = num<P>;
  Sc acc = Sc(0.0);
  const uint2* op = reinterpret_cast<const uint2*>(G.ops) + g.lane;
  const int steps = G.blocks * kProgBlock;
  const uint2 idle = make_uint2(0u, (GF_IDLE << 16) | DST_NONE);
  uint2 n1 = steps > 0 ? __ldg(op) : idle, n2 = steps > 1 ? __ldg(op + g.size) : idle;
#pragma unroll 1
  for (int st = 0; st < steps; ++st) {
    const GatherOp o = as_gop(n1);
    n1 = n2;
    if (st + 2 < steps) n2 = __ldg(op + (size_t)(st + 2) * g.size);
    if (!(o.flags & GF_IDLE)) acc += fin(ld(o.a, o.b), (int)o.b);
    if (o.dst != DST_NONE) {
      if (o.dst & PARTIAL_BIT) part[o.dst & 0x7FFF] = acc;
      else if (ADD) out[o.dst] += acc;
      else out[o.dst] = acc;
      acc = Sc(0.0);
    }
  }
}
template <bool ADD, class P, class PP, class Ld, class Fin, class Gp, class GT>
__device__ __forceinline__ void run_gather(const GT& G, P out, PP part, Ld ld, Fin fin, const Gp& g) {
  using Sc = num<P>;
  if constexpr (is_real<Sc>()) gather_blocks<ADD>(G, out, part, ld, fin, g);
  else gather_steps<ADD>(G, out, part, ld, fin, g);
  g.sync();
  for (int c = g.lane; c < G.n_comb; c += g.size) {
    const int dst = __ldg(G.comb + 3 * c), f = __ldg(G.comb + 3 * c + 1), cnt = __ldg(G.comb + 3 * c + 2);
    Sc s = part[f];
    for (int i = 1; i < cnt; ++i) s += part[f + i];
    if (ADD) out[dst] += s; else out[dst] = s;
  }
  g.sync();
}
// sum of nu x[a] (b encodes nu), and of x[a] y[b]
template <bool ADD, class P, class PP, class Q, class Gp, class GT>
__device__ __forceinline__ void gather_nu(const GT& G, P out, PP part, Q x, const Gp& g) {
  using Sc = num<P>;
  run_gather<ADD>(G, out, part, [&](int a, int) { return Sc(x[a]); }, [](const Sc& v, int b) { return nu_of(b) * v; },
                  g);
}
template <class T1, class T2>
struct Pair {
  T1 x;
  T2 y;
};
template <class P, class PP, class Q1, class Q2, class Gp, class GT>
__device__ __forceinline__ void gather_xy(const GT& G, P out, PP part, Q1 x, Q2 y, const Gp& g) {
  using Pr = Pair<num<Q1>, num<Q2>>;
  run_gather<false>(G, out, part, [&](int a, int b) { return Pr{x[a], y[b]}; },
                    [](const Pr& v, int) { return v.x * v.y; }, g);
}

// -------------------------------------------------------------------------------------- thermo
// One species at T: cp/R, h/RT, g = h/RT - s/R and its exponential (NASA-7, range by T vs T_mid).
template <class Sc>
struct SpOut {
  Sc cpR, hRT, eg, emg, yw, dcp;
};

template <class Sc, class MV, class Q>
__device__ __forceinline__ SpOut<Sc> species_item(const MV& M, int k, double tmid, Q y, Sc T, Sc lnT, Sc invT,
                                                  int tj, double ttau, bool deriv) {
  const double* t = M.sp + k;
  const double iw = __ldg(t);
  const double* cb = t + (size_t)(4 + (less_pos(val(T), tmid) ? 0 : SP_RANGE)) * M.n;
  auto c = [&](int f) { return __ldg(cb + f * M.n); };
  const Sc a0 = c(0), a1 = c(1), a2 = c(2), a3 = c(3), a4 = c(4);
  SpOut<Sc> o;
  o.cpR = sfma(T, sfma(T, sfma(T, sfma(T, a4, a3), a2), a1), a0);
  const Sc h = sfma(T, sfma(T, sfma(T, sfma(T, Sc(c(8)), Sc(c(7))), Sc(c(6))), Sc(c(5))), a0);
  const Sc a5 = c(13), a6 = c(14);
  o.hRT = sfma(a5, invT, h);
  const Sc gp = sfma(T, sfma(T, sfma(T, sfma(T, Sc(c(12)), Sc(c(11))), Sc(c(10))), Sc(c(9))), sfma(a5, invT, -a6));
  bool tabd = false;
  if constexpr (is_real<Sc>()) {
    if (tj >= 0 && M.tab_deg[0] > 0 && M.tab_deg[1] > 0) {
      o.eg = tab_poly(M.tab[0] + ((size_t)tj * M.n + k) * (M.tab_deg[0] + 1), M.tab_deg[0], ttau);
      o.emg = tab_poly(M.tab[1] + ((size_t)tj * M.n + k) * (M.tab_deg[1] + 1), M.tab_deg[1], ttau);
      tabd = true;
    }
  }
  if (!tabd) {
    o.eg = sexp(sfma(a0, 1.0 - lnT, gp));
    o.emg = srcp(o.eg);
  }
  o.yw = y[1 + k] * iw;
  o.dcp = Sc(0.0);
  if (deriv) o.dcp = sfma(T, sfma(T, Sc(c(17)) * T + Sc(c(16)), Sc(c(15))), a1);
  return o;
}

// NASA-7 at T for every species, one species per lane at a time; fills C, hRT, eg = exp(g), emg = 1/eg, cpR.
// A lane's consecutive species enter the sum of Y/W in pairs (first the pair, then the running sum).
template <class P, class Q, class Gp, class MV, class LT>
__device__ __forceinline__ ScalT<num<P>> eval_species(const MV& M, P s, const LT& L, Q y, double p, const Gp& g,
                                                      bool deriv) {
  using Sc = num<P>;
  ScalT<Sc> sc;
  sc.T = y[0];
  sc.lnT = slog(sc.T);
  sc.invT = srcp(sc.T);
  sc.tj = -1;
  sc.ttau = 0.0;
  if constexpr (is_real<Sc>()) tab_locate(M, sc.T, sc.invT, sc.tj, sc.ttau);
  const Sc T = sc.T;
  Sc sig = Sc(0.0), cps = Sc(0.0), dcps = Sc(0.0), first = Sc(0.0);
  bool odd = false;
  const auto hRT = s + L.hRT;
  const auto egv = s + L.eg;
  const auto emg = s + L.emg;
  const auto cpv = s + L.cpR;
  const auto C = s + L.C;
  double tmid = __ldg(M.sp + 2 * M.n + min(g.lane, M.n - 1));   // the range decides which coefficients to read
#pragma unroll 1
  for (int k = g.lane; k < M.n; k += g.size) {
    const double tm = tmid;
    tmid = __ldg(M.sp + 2 * M.n + min(k + g.size, M.n - 1));
    const SpOut<Sc> a = species_item<Sc>(M, k, tm, y, T, sc.lnT, sc.invT, sc.tj, sc.ttau, deriv);
    if (odd) sig += first + a.yw;
    else first = a.yw;
    odd = !odd;
    cps = sfma(a.yw, a.cpR, cps);
    if (deriv) dcps = sfma(a.yw, a.dcp, dcps);
    hRT[k] = a.hRT; egv[k] = a.eg; emg[k] = a.emg; cpv[k] = a.cpR; C[k] = a.yw;
  }
  if (odd) sig += first;
  if (deriv) gsum3(g, sig, cps, dcps);
  else gsum2(g, sig, cps);
  sc.Wbar = srcp(sig);
  sc.ctot = p * sc.invT * (1.0 / kRu);
  sc.rho = sc.ctot * sc.Wbar;
  sc.irho = srcp(sc.rho);
  sc.cp = kRu * cps;
  sc.dcps = dcps;
  sc.rtp = kRu * T * (1.0 / kP0);
  sc.irtp = srcp(sc.rtp);
  g.sync();
  for (int k = g.lane; k < M.n; k += g.size) C[k] *= sc.rho;
  g.sync();
  return sc;
}

// -------------------------------------------------------------------------------------- reactions
// What the rate of progress of one reaction reads besides the cell's own vectors: its record and the
// Arrhenius parameters of the (high-pressure) forward rate.
struct RxIn {
  RxRec i;
  double lnA, b, Ta;
};

template <class MV>
__device__ __forceinline__ RxIn ld_rx(const MV& M, int r) {
  RxIn x;
  const uint4 v = __ldg(reinterpret_cast<const uint4*>(M.rxr + r));
  x.i.r01 = v.x; x.i.r2p0 = v.y; x.i.p12 = v.z; x.i.flags = v.w;
  x.lnA = __ldg(M.rxd + r); x.b = __ldg(M.rxd + M.R + r); x.Ta = __ldg(M.rxd + 2 * M.R + r);
  return x;
}

// Forward rate coefficient (the high-pressure limit of a fall-off reaction) and its logarithm.
template <class Sc, class MV>
__device__ __forceinline__ Sc rx_kf(const MV& M, int r, const RxIn& x, const ScalT<Sc>& sc, Sc& lnk) {
  lnk = sfma(-Sc(x.Ta), sc.invT, sfma(Sc(x.b), sc.lnT, Sc(x.lnA)));
  if constexpr (is_real<Sc>()) {
    if (sc.tj >= 0 && M.tab_deg[2] > 0)
      return tab_poly(M.tab[2] + ((size_t)sc.tj * M.R + r) * (M.tab_deg[2] + 1), M.tab_deg[2], sc.ttau);
  }
  return sexp(lnk);
}

// A simple reaction (RXF_SIMPLE: A + B <=> C + D, four different species, no third body), which most reactions
// of a mechanism are.  The same operations in the same order as rx_core / rx_store with those counts, without
// the factors that are 1 and the terms that are 0 there: 19 FP64 instructions instead of 28 for the rate of
// progress, and 34 instead of about 75 with the derivatives (dq/dT into s[dq_off + r], the four slots dq/dC
// from s[d_off + so] on).  The FP64 pipe takes one warp instruction per 64 cycles and is what bounds this code:
// with it and the tables as structures of arrays, the source term of 65,536 cells of 53 species / 325 reactions
// went from 2999 to 2667 us, the Jacobian of 8,191 cells from 1236 to 1071 us.
template <class Sc, class P, class MV, class LT, class Sink>
__device__ __forceinline__ void rx_simple(const MV& M, int r, const RxIn& in, P s, const LT& L, const ScalT<Sc>& sc,
                                          bool valid, bool deriv, Sink& to) {
  const int r0 = in.i.r01 & 0xffff, r1 = in.i.r01 >> 16, p0 = in.i.r2p0 >> 16, p1 = in.i.p12 & 0xffff;
  const auto C = s + L.C, eg = s + L.eg, emg = s + L.emg;
  Sc lnk;
  const Sc kf = rx_kf(M, r, in, sc, lnk);
  const Sc cr0 = C[r0], cr1 = C[r1], cp0 = C[p0], cp1 = C[p1];
  Sc ik = Sc(eg[p0]) * Sc(emg[r0]);
  ik *= Sc(eg[p1]);
  ik *= Sc(emg[r1]);
  const Sc kr = kf * ik;
  const Sc q = sfma(kf, cr0 * cr1, -(kr * (cp0 * cp1)));
  if (valid) to.rate(r, in.i, q);
  if (deriv) {
    const auto hRT = s + L.hRT;
    const int so = (int)(in.i.flags >> 16);
    const Sc dlnkf = sfma(Sc(in.Ta), sc.invT, Sc(in.b)) * sc.invT;
    Sc sh = Sc(hRT[p0]) - Sc(hRT[r0]);
    sh += Sc(hRT[p1]);
    sh -= Sc(hRT[r1]);
    const Sc dlnKc = smul(sh, sc.invT);
    Sc s0 = kf * cr1, s1 = kf * cr0, s2 = kr * cp1, s3 = kr * cp0;
    const Sc qf = s1 * cr1, qr = s3 * cp1;
    Sc dq = sfma(dlnkf, qf, -((dlnkf - dlnKc) * qr));
    s2 = -s2;
    s3 = -s3;
    if (!finite_bits(val(kf)) || !finite_bits(val(kr)) || !finite_bits(val(sc.ctot)) || !finite_bits(val(sc.invT))) {
      // the zero terms are not neutral next to infinities and NaN
      s0 = sfma(-kr, Sc(0.0), s0); s1 = sfma(-kr, Sc(0.0), s1);
      s2 = sfma(kf, Sc(0.0), s2); s3 = sfma(kf, Sc(0.0), s3);
      dq = dq - Sc(0.0) * sc.ctot * sc.invT;
    }
    if (valid) {
      to.dT(r, dq);
      to.slot(so, s0); to.slot(so + 1, s1); to.slot(so + 2, s2); to.slot(so + 3, s3);
    }
  }
}

// Table records of listed colliders and derivative slots are read in batches (one by one for dual numbers): each read is a trip to L2, and
// one after the other they took as long as the reaction's exponentials.
template <class Sc>
__host__ __device__ constexpr int batch_of() { return is_real<Sc>() ? 4 : 1; }
__device__ __forceinline__ EffRec ld_rec(const EffRec* p) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(p));
  return EffRec{__hiloint2double(v.y, v.x), v.z, 0};
}
__device__ __forceinline__ SlotRec ld_rec(const SlotRec* p) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(p));
  return SlotRec{__hiloint2double(v.y, v.x), v.z, 0};
}

// Per-reaction quantities of the rate evaluation that the derivative part needs afterwards.
template <class Sc>
struct RxCore {
  Sc q, qn, kf, kr, Mfac, dlnkf_dT, dlnKc_dT, dlnk_dlnM, iM;
  Sc cr0, cr1, cr2, cp0, cp1, cp2;
  int so, scn;
};

// Rate of progress of reaction r of any type (0 elementary, 1 third-body, 2 Troe).  Branch-free in the participant
// counts: absent occurrences read index 0 and count as 1.
template <class Sc, class P, class MV>
__device__ __forceinline__ RxCore<Sc> rx_core(const MV& M, int r, int type, const RxIn& in, P C, P eg, P emg, P hRT,
                                              const ScalT<Sc>& sc, bool deriv) {
  // everything that is read from the tables is asked for before the first exponential
  int4 w = make_int4(0, 0, 0, 0);   // efficiency count, slot offset, slot count, efficiency offset
  if (type != 0 || deriv) w = __ldg(reinterpret_cast<const int4*>(M.rxi + (size_t)r * RX_I) + 3);
  double par[11];
  if (type == 2) {
#pragma unroll
    for (int f = 3; f < 11; ++f) par[f] = __ldg(M.rxd + r + f * M.R);
  }
  const int rev = in.i.flags & RXF_REV, nro = (in.i.flags >> 1) & 3, npo = (in.i.flags >> 3) & 3;
  const int r0 = in.i.r01 & 0xffff, r1 = in.i.r01 >> 16, r2 = in.i.r2p0 & 0xffff;
  const int p0 = in.i.r2p0 >> 16, p1 = in.i.p12 & 0xffff, p2 = in.i.p12 >> 16;
  const Sc bb = in.b, Ta = in.Ta;
  RxCore<Sc> x;
  Sc lnkinf;
  Sc kf = rx_kf(M, r, in, sc, lnkinf);
  auto at = [](P v, bool there, int i, double other) { return there ? Sc(v[i]) : Sc(other); };
  x.cr0 = C[r0]; x.cr1 = at(C, nro > 1, r1, 1.0); x.cr2 = at(C, nro > 2, r2, 1.0);
  x.cp0 = C[p0]; x.cp1 = at(C, npo > 1, p1, 1.0); x.cp2 = at(C, npo > 2, p2, 1.0);
  const Sc Pf = x.cr0 * x.cr1 * x.cr2, Pb = x.cp0 * x.cp1 * x.cp2;
  Sc Mv = sc.ctot;
  if (type != 0) {
    constexpr int kBatch = batch_of<Sc>();
    for (int i = 0; i < w.x; i += kBatch) {   // a batch of listed colliders is read at once
      EffRec e[kBatch];
#pragma unroll
      for (int j = 0; j < kBatch; ++j) e[j] = ld_rec(M.eff + w.w + min(i + j, w.x - 1));
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const Sc c = C[e[j].sp];
        if (i + j < w.x) Mv = sfma(Sc(e[j].am1), c, Mv);
      }
    }
  }
  x.dlnkf_dT = Sc(0.0);
  if (deriv) x.dlnkf_dT = sfma(Ta, sc.invT, bb) * sc.invT;
  x.dlnk_dlnM = Sc(0.0);
  x.iM = Sc(0.0);
  if (type == 2) {
    const Sc lnk0 = sfma(-Sc(par[5]), sc.invT, sfma(Sc(par[4]), sc.lnT, Sc(par[3])));
    const Sc lnM = slog(Mv);
    const Sc lnPr = lnk0 - lnkinf + lnM;
    const Sc Pr = sexp(lnPr);
    const double T2 = par[10];
    // the Troe centre: tabulated (Troe reactions are the first compiled ones), or from its three
    // exponentials, which the Jacobian's temperature derivative needs in any case
    bool tfc = false;
    if constexpr (is_real<Sc>()) tfc = sc.tj >= 0 && M.tab_deg[3] > 0;
    Sc e3 = Sc(0.0), e1 = Sc(0.0), e2 = Sc(0.0), Fc;
    if (!tfc || deriv) {
      e3 = sexp(-sc.T * par[8]);
      e1 = sexp(-sc.T * par[9]);
      e2 = less_pos(0.0, T2) ? sexp(-T2 * sc.invT) : Sc(0.0);
    }
    if constexpr (is_real<Sc>()) {
      if (tfc) Fc = tab_poly(M.tab[3] + ((size_t)sc.tj * M.n_troe + r) * (M.tab_deg[3] + 1), M.tab_deg[3], sc.ttau);
    }
    if (!tfc) Fc = sfma(Sc(par[6]), e3, sfma(Sc(par[7]), e1, e2));
    const Sc Lc = slog(Fc) * kInvLn10;
    const Sc cc = sfma(Sc(-0.67), Lc, Sc(-0.4));
    const Sc nn = sfma(Sc(-1.27), Lc, Sc(0.75));
    const Sc xx = sfma(lnPr, Sc(kInvLn10), cc);
    const Sc den = sfma(Sc(-0.14), xx, nn);
    // three reciprocals from one division: 1/den, 1/(1 + f1^2) = den^2/S2 with S2 = den^2 + xx^2, and
    // 1/(1 + Pr), all from R = 1/(den S2 (1 + Pr))
    const Sc pr1 = 1.0 + Pr;
    const Sc S2 = sfma(xx, xx, den * den);
    const Sc dp = den * pr1;
    const Sc R = srcp(dp * S2);
    const Sc iden = S2 * pr1 * R;
    const Sc f1 = xx * iden;
    const Sc ib = den * dp * R * den;
    const Sc F = sexp(Lc * ib * kLn10);
    const Sc ipr1 = den * S2 * R;
    kf = kf * (Pr * ipr1) * F;
    if (deriv) {
      const Sc dlnk0_dT = sfma(Sc(par[5]), sc.invT, Sc(par[4])) * sc.invT;
      const Sc dlnPr_dT = dlnk0_dT - x.dlnkf_dT;
      const Sc dFc_dT = -(par[6] * par[8]) * e3 - (par[7] * par[9]) * e1 +
                        T2 * sc.invT * sc.invT * e2;
      const Sc dLc_dT = dFc_dT / Fc * kInvLn10;
      const Sc dx_dT = sfma(dlnPr_dT, Sc(kInvLn10), -0.67 * dLc_dT);
      const Sc dnn_dT = -1.27 * dLc_dT;
      const Sc df1_dT = (dx_dT * nn - xx * dnn_dT) * iden * iden;
      const Sc dlog10F_dT = sfma(dLc_dT, ib, -2.0 * Lc * f1 * df1_dT * ib * ib);
      x.dlnkf_dT = x.dlnkf_dT + dlnPr_dT * ipr1 + kLn10 * dlog10F_dT;
      const Sc df1_dlnM = nn * kInvLn10 * iden * iden;
      x.dlnk_dlnM = ipr1 - kLn10 * 2.0 * Lc * f1 * df1_dlnM * ib * ib;
      x.iM = sexp(-lnM);
    }
  }
  // reverse rate: k_r = k_f * prod exp(g)^nu'' * prod exp(-g)^nu' * (Ru T/p0)^(sum nu)
  const int dn = npo - nro;
  Sc ik = Sc(eg[p0]) * Sc(emg[r0]);
  ik *= at(eg, npo > 1, p1, 1.0) * at(eg, npo > 2, p2, 1.0);
  ik *= at(emg, nro > 1, r1, 1.0) * at(emg, nro > 2, r2, 1.0);
  const Sc fp = dn > 0 ? sc.rtp : sc.irtp;
  const int adn = dn < 0 ? -dn : dn;
  ik *= (adn >= 1 ? fp : Sc(1.0)) * (adn >= 2 ? fp : Sc(1.0)) * (adn >= 3 ? fp : Sc(1.0));
  x.kr = rev ? kf * ik : Sc(0.0);
  x.kf = kf;
  if (deriv) {
    Sc sh = Sc(hRT[p0]) - Sc(hRT[r0]);
    sh += at(hRT, npo > 1, p1, 0.0) + at(hRT, npo > 2, p2, 0.0);
    sh -= at(hRT, nro > 1, r1, 0.0) + at(hRT, nro > 2, r2, 0.0);
    const double dnd = dn == 0 ? 0.0 : dn == 1 ? 1.0 : dn == -1 ? -1.0 : dn == 2 ? 2.0 : dn == -2 ? -2.0 :
                       dn == 3 ? 3.0 : -3.0;
    x.dlnKc_dT = rev ? (sh - dnd) * sc.invT : Sc(0.0);
  } else {
    x.dlnKc_dT = Sc(0.0);
  }
  x.Mfac = type == 1 ? Mv : Sc(1.0);
  x.qn = sfma(kf, Pf, -(x.kr * Pb));
  x.q = x.Mfac * x.qn;
  x.so = w.y;
  x.scn = w.z;
  return x;
}

// Store q (and with deriv: dq/dT at fixed C into s[dq_off + r], and the derivative slots dq/dC_j into
// s[d_off + slot]) of reaction r.
template <class Sc, class MV, class Sink>
__device__ __forceinline__ void rx_store(const MV& M, int r, int type, const RxRec& rec, const RxCore<Sc>& x,
                                         const ScalT<Sc>& sc, bool valid, bool deriv, Sink& to) {
  if (!valid) return;
  to.rate(r, rec, x.q);
  if (!deriv) return;
  const Sc kfM = x.kf * x.Mfac, krM = x.kr * x.Mfac;
  const Sc qf = kfM * x.cr0 * x.cr1 * x.cr2, qr = krM * x.cp0 * x.cp1 * x.cp2;
  Sc dqdM = Sc(0.0);
  if (type == 1) dqdM = x.qn;
  if (type == 2) dqdM = x.dlnk_dlnM * x.q * x.iM;
  // [M] depends on T through the total concentration p/(Ru T)
  to.dT(r, sfma(x.dlnkf_dT, qf, -((x.dlnkf_dT - x.dlnKc_dT) * qr)) - dqdM * sc.ctot * sc.invT);
  // partial products: d(prod)/d(occurrence i) = product of the other occurrences
  const Sc dr0 = x.cr1 * x.cr2, dr1 = x.cr0 * x.cr2, dr2 = x.cr0 * x.cr1;
  const Sc dp0 = x.cp1 * x.cp2, dp1 = x.cp0 * x.cp2, dp2 = x.cp0 * x.cp1;
  const bool fin = finite_bits(val(kfM)) && finite_bits(val(krM));
  constexpr int kBatch = batch_of<Sc>();
  for (int i0 = 0; i0 < x.scn; i0 += kBatch) {
    SlotRec slots[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) slots[j] = ld_rec(M.dslot + x.so + min(i0 + j, x.scn - 1));
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const int i = i0 + j, mask = slots[j].mask;
      if (i >= x.scn) break;
      // elementary reactions list no colliders: their (efficiency - 1) is 0 and so is the [M] term
      Sc v = type == 0 ? Sc(0.0) : slots[j].am1 * dqdM;
      if (mask != 0 || !fin) {   // a participant (a species that only collides has no factor: the [M] term is all)
        // the slot's factor on a side is the sum over the species' occurrences there, nearly always one: it is
        // selected, and a second or third one added
        Sc fr = (mask & 1) ? dr0 : (mask & 2) ? dr1 : (mask & 4) ? dr2 : Sc(0.0);
        Sc fq = (mask & 8) ? dp0 : (mask & 16) ? dp1 : (mask & 32) ? dp2 : Sc(0.0);
        if ((mask & 3) == 3 || (mask & 5) == 5 || (mask & 6) == 6) {
          if ((mask & 3) == 3) fr += dr1;
          if ((mask & 4) && (mask & 3)) fr += dr2;
        }
        if ((mask & 24) == 24 || (mask & 40) == 40 || (mask & 48) == 48) {
          if ((mask & 24) == 24) fq += dp1;
          if ((mask & 32) && (mask & 24)) fq += dp2;
        }
        v = sfma(kfM, fr, v);
        v = sfma(-krM, fq, v);
      }
      to.slot(x.so + i, v);
    }
  }
}

// Where eval_reactions leaves its results: q, and with derivatives dq/dT and the slots, in the cell's memory.
template <class P>
struct ToCell {
  P s;
  int q_off, dq_off, d_off;
  __device__ __forceinline__ void rate(int r, const RxRec&, const num<P>& q) const { s[q_off + r] = q; }
  __device__ __forceinline__ void dT(int r, const num<P>& v) const { s[dq_off + r] = v; }
  __device__ __forceinline__ void slot(int i, const num<P>& v) const { s[d_off + i] = v; }
};

// Rates of progress of reactions [rb, re), in rounds of one reaction per lane; to.rate(), and with deriv to.dT() and
// to.slot(), take each reaction's results.  A round whose reactions are all simple takes the short form (every lane
// of a round's warp takes part: lanes past the end repeat the last reaction and leave nothing).  The other types
// stand first (Troe, third-body) and share their rounds: what a Troe or third-body reaction needs beyond an
// elementary one is a branch that the round takes once.
template <class Sc, class P, class Gp, class MV, class LT, class Sink>
__device__ __forceinline__ void eval_reactions(const MV& M, P s, const LT& L, const ScalT<Sc>& sc,
                                               const Gp& g, int rb, int re, bool deriv, Sink& to) {
  const auto C = s + L.C, eg = s + L.eg, emg = s + L.emg, hRT = s + L.hRT;
  if (rb < re) {
    RxIn next = ld_rx(M, min(rb + g.lane, re - 1));
#pragma unroll 1
    for (int base = rb; base < re; base += g.size) {
      const int r = min(base + g.lane, re - 1);
      const bool valid = base + g.lane < re;
      const RxIn in = next;
      if (base + g.size < re) next = ld_rx(M, min(base + g.size + g.lane, re - 1));
      if (wall(g, (in.i.flags & RXF_SIMPLE) != 0)) {
        rx_simple<Sc>(M, r, in, s, L, sc, valid, deriv, to);
      } else {
        const int type = r < M.n_troe ? 2 : r < M.n_troe + M.n_tb ? 1 : 0;
        rx_store<Sc>(M, r, type, in.i, rx_core<Sc>(M, r, type, in, C, eg, emg, hRT, sc, deriv), sc, valid, deriv, to);
      }
    }
  }
  g.sync();
}

// One pass over the reactions (all of them in one for a right-hand side; for the Jacobian those whose slots fit).
template <class MV, class P, class LT, class Sc, class Gp>
__device__ __forceinline__ void eval_pass(const MV& M, P s, const LT& L, const ScalT<Sc>& sc, const Gp& g, int ps,
                                          bool deriv) {
  const int rb = deriv ? M.jpass[ps][JP_RB] : 0, re = deriv ? M.jpass[ps][JP_RE] : M.R;
  const int cnt = M.jpass[ps][JP_CNT];
  const ToCell<P> to{s, L.q, L.D - rb, L.D + cnt - M.jpass[ps][JP_SB]};
  eval_reactions<Sc>(M, s, L, sc, g, rb, re, deriv, to);
}

// ---- helper warps.  With few cells a call takes as long as its longest cell's chain of attempts, and the chip is not
// full.  Then a block holds one cell of one or two warps and some helper warps, which take their shares of its reaction
// rounds and wait at their common barrier for the rest of the time.  A reaction's results don't depend on the lane that
// evaluates it, and sums and programs stay with the cell's own lanes, so the results are bit for bit those without the
// helpers.  53 species / 325 reactions: the 11 rounds of a rate evaluation become 3 with three helpers, 6 with one; a
// 10 us call takes 108 ms instead of 131 at 304 cells and 144 instead of 165 at 456 (RODAS4, 300 cells: 55 instead of
// 71).  150 / 1000: with two helpers for a cell of two warps 255 ms instead of 284 at 100 cells, with three for a cell
// of one warp 290 instead of 378 at 300.
struct HelpOrder {   // what the helpers need to know besides the cell's memory
  Scal sc;
  int ps, deriv, more;   // more = 0: the cell's own warps have ended
};
__device__ __forceinline__ HelpOrder& help_order() {
  __shared__ HelpOrder order;
  return order;
}
// A cell's own lanes and its helpers.  They meet at a named barrier with their number spelt out, because they come to it
// from different places (the helpers from their loop, the cell's warps from its rate evaluations), which
// __syncthreads() does not allow for.  (Barrier 0 is __syncthreads(), 1 a two-warp cell's own.)
template <class Gp, int H>
struct GrpHelp {
  static constexpr int size = Gp::size + H * kWarp;
  static constexpr int bar = 2;
  int lane;
  __device__ __forceinline__ void sync() const {
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"n"(bar), "n"(size) : "memory");
  }
};
template <class Gp, int H>
__device__ __forceinline__ bool wall(const GrpHelp<Gp, H>&, bool ok) { return __all_sync(0xffffffffu, ok); }
template <class Gp, class MV, class LT>
__device__ __forceinline__ void help(const MV& M, double* s, const LT& L) {
  const HelpOrder& o = help_order();
  const GrpHelp<Gp, MV::kHelpers> g{(int)threadIdx.x};
#pragma unroll 1
  while (true) {
    g.sync();
    if (!o.more) return;
    const Scal sc = o.sc;
    eval_pass(M, s, L, sc, g, o.ps, o.deriv != 0);   // ends with a barrier of the group
  }
}
template <class Gp, int H>
__device__ __forceinline__ void help_end() {
  if (threadIdx.x == 0) help_order().more = 0;
  GrpHelp<Gp, H>{(int)threadIdx.x}.sync();
}

// -------------------------------------------------------------------------------------- f and J
// The rates at y: C, h/RT, the rates of progress q and the production rates w_k into w[n].  With deriv also the
// Y block of S (Dtil) and w_T in the T-column slots of S.  For those the reactions run in passes (see
// MechView::jpass): each pass leaves dq/dT and the derivative slots of its reactions in the region D, and its
// gather adds them into S.  deriv is a run-time flag so that a kernel that needs both holds the code once.
template <class P, class Q, class W, class Gp, class MV, class LT>
__device__ __forceinline__ ScalT<num<P>> eval_rates(const MV& M, P s, const LT& L, Q y, double p, W w, const Gp& g,
                                                    bool deriv) {
  using Sc = num<P>;
  const ScalT<Sc> sc = eval_species(M, s, L, y, p, g, deriv);
  const auto S = s + L.S;
  const auto sp = prog_ptr(s);
  if (deriv)
    for (int e = g.lane; e < M.nY + M.n; e += g.size) S[e] = Sc(0.0);
  const int passes = deriv ? M.n_jpass : 1;
#pragma unroll 1
  for (int ps = 0; ps < passes; ++ps) {
    if constexpr (MV::kHelpers > 0) {
      if (g.lane == 0) {
        HelpOrder& o = help_order();
        if (ps == 0) o.sc = sc;
        o.ps = ps;
        o.deriv = deriv;
        o.more = 1;
      }
      const GrpHelp<Gp, MV::kHelpers> all{g.lane};
      all.sync();
      eval_pass(M, s, L, sc, all, ps, deriv);
    } else {
      eval_pass(M, s, L, sc, g, ps, deriv);
    }
    if (deriv && ps == 0) gather_nu<false>(M.g_jac[0], sp + L.S, sp + L.part, sp + L.D, g);
    if (deriv && ps > 0) gather_nu<true>(M.g_jac[ps], sp + L.S, sp + L.part, sp + L.D, g);
  }
  gather_nu<false>(M.g_omega, prog_ptr(w), sp + L.part, sp + L.q, g);
  return sc;
}

// f from the production rates, in place: out[1 + k] holds w_k on entry.
template <class Sc, class P, class Gp, class MV, class LT>
__device__ __forceinline__ void finish_f(const MV& M, P s, const LT& L, const ScalT<Sc>& sc, P out, const Gp& g) {
  const P w = out + 1;
  Sc Qs = Sc(0.0);
  for (int k = g.lane; k < M.n; k += g.size) {
    const Sc om = w[k];
    Qs = sfma(Sc(s[L.hRT + k]), om, Qs);
    w[k] = om * __ldg(M.sp + M.n + k) * sc.irho;
  }
  Qs = gsum(g, Qs);
  if (g.lane == 0) out[0] = sdiv(-kRu * sc.T * Qs, sc.rho * sc.cp);
  g.sync();
}

// f(y) into out[m].  Uses C/hRT/eg/emg/cpR/q scratch.  Returns the scalars of the evaluation.
template <class P, class Q, class Gp, class MV, class LT>
__device__ __forceinline__ ScalT<num<P>> eval_f(const MV& M, P s, const LT& L, Q y, double p, P out, const Gp& g) {
  const ScalT<num<P>> sc = eval_rates(M, s, L, y, p, out + 1, g, false);
  finish_f(M, s, L, sc, out, g);
  return sc;
}

// f(y) into f0[m], S[nnz_S] (internal order), u[m], v[m] from what eval_rates with deriv left: w_k in x, Dtil and
// w_T in S (the T column takes w_T's place).  Scratch: U1 (g), U2 (t).
template <class Sc, class P, class Gp, class MV, class LT>
__device__ __forceinline__ void finish_jac(const MV& M, P s, const LT& L, const ScalT<Sc>& sc, const Gp& g) {
  const auto w = s + L.x, gk = s + L.U1, tk = s + L.U2, S = s + L.S, wT = s + (L.S + M.nY);
  const auto C = s + L.C, hRT = s + L.hRT;
  const auto sp = prog_ptr(s);
  // the tables of the loops below are asked for ahead of the sums before them
  const int k0 = min(g.lane, M.n - 1);
  double nW = __ldg(M.sp + M.n + k0), niW = __ldg(M.sp + k0);
  gather_xy(M.g_row, sp + L.U1, sp + L.part, sp + L.S, sp + L.C, g);
  gather_xy(M.g_col, sp + L.U2, sp + L.part, sp + L.S, sp + L.hRT, g);
  const auto f = s + L.f0, u = s + L.u, v = s + L.v;
  const Sc T = sc.T;
  // f, u and the T column; partial sums for the T row scalars
  Sc Qs = Sc(0.0), A1 = Sc(0.0), A2 = Sc(0.0);
  for (int k = g.lane; k < M.n; k += g.size) {
    const double Wk = nW, iWk = niW;
    const int kn = min(k + g.size, M.n - 1);
    nW = __ldg(M.sp + M.n + kn);
    niW = __ldg(M.sp + kn);
    const Sc om = w[k], g = gk[k];
    const Sc dwT = sfma(-g, sc.invT, Sc(wT[k]));   // read before the T column overwrites w_T
    const Sc fk = Wk * om * sc.irho;
    f[1 + k] = fk;
    u[1 + k] = Wk * sc.irho * (om - g);
    S[M.nY + k] = sfma(Wk * sc.irho, dwT, fk * sc.invT);
    v[1 + k] = sc.Wbar * iWk;
    const Sc h = hRT[k];
    Qs = sfma(h, om, Qs);
    A1 = sfma(Sc(s[L.cpR + k]), om, sfma(T * h, dwT, A1));
    A2 = sfma(h, g, A2);
  }
  constexpr int kScale = 8;   // the first batch of the species block's factors
  double ratio[kScale];
#pragma unroll
  for (int i = 0; i < kScale; ++i) ratio[i] = __ldg(M.entry_wratio + min(g.lane + i * g.size, M.nY - 1));
  gsum3(g, Qs, A1, A2);
  const Sc rcp = sc.rho * sc.cp;
  const Sc fT = sdiv(-kRu * T * Qs, rcp);
  // T row: S_Tj for species j, then S_TT; u_T; v_T
  for (int j = g.lane; j < M.n; j += g.size) {
    const double iw = __ldg(M.sp + j);
    S[M.nY + M.n + 1 + j] = sdiv(-kRu * sfma(T, Sc(tk[j]), fT * Sc(s[L.cpR + j])) * iw, sc.cp);
  }
  if (g.lane == 0) {
    f[0] = fT;
    S[M.nY + M.n] = sdiv(-kRu * A1, rcp) + fT * (sc.invT - sdiv(kRu * sc.dcps, sc.cp));
    u[0] = sdiv(kRu * T * A2, rcp) + fT;
    v[0] = Sc(0.0);
  }
  g.sync();
  // species block: S_kj = (W_k / W_j) Dtil_kj (after the row and column sums used Dtil)
  for (int e0 = 0; e0 < M.nY; e0 += kScale * g.size) {
#pragma unroll
    for (int i = 0; i < kScale; ++i) {
      const int e = e0 + g.lane + i * g.size;
      if (e < M.nY) S[e] *= ratio[i];
      ratio[i] = __ldg(M.entry_wratio + min(e + kScale * g.size, M.nY - 1));
    }
  }
  g.sync();
}

// f(y) into f0[m], S[nnz_S] (internal order), u[m], v[m].  Scratch: C.., q, the pass region D, x, U1, U2.
template <class P, class Q, class Gp, class MV, class LT>
__device__ __forceinline__ ScalT<num<P>> eval_jac(const MV& M, P s, const LT& L, Q y, double p, const Gp& g) {
  const ScalT<num<P>> sc = eval_rates(M, s, L, y, p, s + L.x, g, true);
  finish_jac(M, s, L, sc, g);
  return sc;
}

// -------------------------------------------------------------------------------------- linear algebra
// LU of A = I/(h gamma) - S, in place, by the precomputed elimination program.  false if a pivot is 0
// or not finite.
template <class Gp, class MV, class LT>
__device__ __forceinline__ bool lu_build_factor(const MV& M, SPtr s, const LT& L, double gh,
                                                const Gp& g) {
  const SPtr LU = s + L.LU;   // followed by the negated reciprocal pivots (L.dinv)
  const SPtr S = s + L.S;
#pragma unroll 8
  for (int l = g.lane; l < M.nnz_LU; l += g.size) {
    const int src = __ldg(M.lu_src + l);
    const double v = S[max(src, 0)];
    LU[l] = src >= 0 ? -v : 0.0;
  }
  g.sync();
  for (int i = g.lane; i < M.m; i += g.size) LU[__ldg(M.lu_diag + i)] += gh;
  g.sync();
  return gall(g, run_fma<true>(M.lu, LU, LU, g.lane, g.size, g));
}

// x <- A^{-1} x (forward and backward substitution by the precomputed program; state-order vector).
template <class Gp, class MV, class LT>
__device__ __forceinline__ void lu_solve(const MV& M, SPtr s, const LT& L, SPtr x, const Gp& g) {
  run_fma<false>(M.sv, s + L.LU, x, g.lane, g.size, g);
}

// The same for two right-hand sides: half of the group's lanes take each (a step of the program has about ten ops,
// so half the lanes need few more steps, and an FP64 instruction costs the same for 16 lanes as for 32).
template <class Gp, class MV, class LT>
__device__ __forceinline__ void lu_solve2(const MV& M, SPtr s, const LT& L, SPtr x1, SPtr x2, const Gp& g) {
  constexpr int half = Gp::size / 2;
  const bool second = g.lane >= half;
  run_fma<false>(M.sv2, s + L.LU, second ? x2 : x1, second ? g.lane - half : g.lane, half, half_sync(g));
  g.sync();
}

// x <- M^{-1} x with M = A - u v^T:  x = A^-1 x + z (v . A^-1 x) / (1 - v . z),  z = A^-1 u
template <class Gp, class MV, class LT>
__device__ __forceinline__ void sm_solve(const MV& M, SPtr s, const LT& L, SPtr x, double iden, const Gp& g) {
  lu_solve(M, s, L, x, g);
  const SPtr v = s + L.v, z = s + L.z;
  double d = 0.0;
  for (int i = g.lane; i < M.m; i += g.size) d = fma(v[i], x[i], d);
  d = gsum(g, d) * iden;
  for (int i = g.lane; i < M.m; i += g.size) x[i] = fma(z[i], d, x[i]);
  g.sync();
}

// -------------------------------------------------------------------------------------- step
struct StepOut {
  bool good;
  double err;
};

// One attempt of size h from y with method 0 RODAS3, 1 ROS2 or 2 RODAS4; need_jac: f0, S, u, v are evaluated at y
// first (otherwise they hold that already), then after_jac sees the evaluation's scalars.  ynew into ytmp, err into the return value.  U1..U4, x, z, LU are
// scratch: RODAS4's U5 lives in the Jacobian's w_k vector (x), its stage 6 gathers the coefficient sum into U1 and
// takes U2's place, both dead by then.
// All stages of all methods, the Jacobian included, go through one loop with one copy of the rates and of the
// solve.  Written out, the kernel held four copies of the rates and nine of the solve and waited on instruction
// fetch.
struct NoHook {
  __device__ __forceinline__ void operator()(const Scal&) const {}
};
template <class Gp, class MV, class LT, class Hook = NoHook>
__device__ __forceinline__ StepOut ros_attempt(const MV& M, double* sd, const LT& L, double p, double h,
                                               double rtol, double atol, const Gp& g, int method, bool need_jac,
                                               Hook after_jac = Hook()) {
  StepOut so{false, 0.0};
  const int m = M.m;
  const SPtr s = shared_ptr(sd);
  const double ih = rcp_rn(h);
  const SPtr y = s + L.y, yt = s + L.ytmp, f0 = s + L.f0, U1 = s + L.U1, U2 = s + L.U2, z = s + L.z;
  const SPtr u = s + L.u, v = s + L.v;
  // U1..U4 are consecutive vectors, U5 is x
  auto U = [&](int j) { return j < 4 ? U1 + j * (L.U2 - L.U1) : s + L.x; };
  const int stages = method == 0 ? 4 : method == 1 ? 2 : 6;
  double iden = 0.0;
  bool fine = true;   // (the other cell of the warp goes on when this one has failed)
#pragma unroll 1
  for (int k = 0; k < stages; ++k) {   // stage k + 1
    const SPtr out = k == 0 ? s + (L.x - 1) : k < 5 ? U(k) : U2;   // stage 1: the production rates go to x
    const bool rates = k == 0 ? need_jac : (method != 0 || k > 1);   // RODAS3's stage 2 takes f(y) again (a21 = 0)
    if (k > 0 && rates) {
      if (k < 5) {
        for (int i = g.lane; i < m; i += g.size) {
          double acc = y[i];
          for (int j = 0; j < k; ++j) {
            const double a = stage_a(method, k, j);
            if (__double2hiint(a) != 0) acc = fma(a, U(j)[i], acc);
          }
          yt[i] = acc;
        }
      } else {   // RODAS4's stage 6: stage 5's point plus U5; the coefficient sum goes into U1
        for (int i = g.lane; i < m; i += g.size) {
          yt[i] += U(4)[i];
          double acc = kR4C[4][4] * U(4)[i];
          for (int j = 3; j >= 0; --j) acc = fma(kR4C[4][j], U(j)[i], acc);
          U1[i] = ih * acc;
        }
      }
      g.sync();
    }
    if (rates) {
      double* to = sd + (k == 0 ? L.x - 1 : k < 4 ? L.U1 + k * (L.U2 - L.U1) : k == 4 ? L.x : L.U2);
      const Scal sc = eval_rates(M, sd, L, sd + (k == 0 ? L.y : L.ytmp), p, to + 1, g, k == 0);
      if (k == 0) {
        finish_jac(M, sd, L, sc, g);
        after_jac(sc);
      } else {
        finish_f(M, sd, L, sc, to, g);
      }
    }
    if (k == 0) {
      fine = lu_build_factor(M, s, L, ih * (method == 1 ? 1.0 / RG2 : method == 2 ? 1.0 / RG4 : 1.0 / RG), g);
      if (!any_cell(g, fine)) return so;
      // z = A^-1 u (the Sherman-Morrison vector) and stage 1's A^-1 f0 together, then stage 1's correction
      for (int i = g.lane; i < m; i += g.size) { z[i] = u[i]; U1[i] = f0[i]; }
      g.sync();
      lu_solve2(M, s, L, z, U1, g);
      double vz = 0.0, vx = 0.0;
      for (int i = g.lane; i < m; i += g.size) { vz = fma(v[i], z[i], vz); vx = fma(v[i], U1[i], vx); }
      gsum2(g, vz, vx);
      const double den = 1.0 - vz;
      fine = fine && (__double_as_longlong(den) << 1) != 0 && finite_bits(den);
      if (!any_cell(g, fine)) return so;
      iden = rcp_rn(den);
      vx *= iden;
      for (int i = g.lane; i < m; i += g.size) U1[i] = fma(z[i], vx, U1[i]);
      g.sync();
      continue;
    }
    for (int i = g.lane; i < m; i += g.size) {
      const double f = (rates ? out : f0)[i];
      if (k == 1) {
        out[i] = fma(stage_c(method, 1, 0) * ih, U1[i], f);
      } else if (k < 5) {
        int j = k - 2;
        double acc = stage_c(method, k, k - 1) * U(k - 1)[i];
        if (method == 0 && k == 3) {   // c42 = -1: one rounding with the product before it
          acc = fma(C43, U(2)[i], -(double)U(1)[i]);
          j = 0;
        }
        for (; j >= 0; --j) acc = fma(stage_c(method, k, j), U(j)[i], acc);
        out[i] = fma(ih, acc, f);
      } else {
        out[i] = f + U1[i];
      }
    }
    g.sync();
    sm_solve(M, s, L, out, iden, g);
  }
  // solution, embedded error, scaled RMS norm (RODAS3: the error is U4; RODAS4: the solution is stage 6's point plus
  // U6, which is the error)
  const SPtr U3 = U(2), U4 = U(3);
  double e2 = 0.0;
  bool fin = true;
  for (int i = g.lane; i < m; i += g.size) {
    double yn, ei;
    if (method == 0) {
      yn = fma(M4, U4[i], fma(M3, U3[i], fma(M1, U1[i], y[i])));
      ei = U4[i];
    } else if (method == 1) {
      yn = fma(R2_M2, U2[i], fma(R2_M1, U1[i], y[i]));
      ei = R2_E * (U1[i] + U2[i]);
    } else {
      yn = yt[i] + U2[i];
      ei = U2[i];
    }
    yt[i] = yn;
    const double sc = fma(rtol, max_mag(y[i], yn), atol);
    const double e = div_rn(ei, sc);
    e2 = fma(e, e, e2);
    fin = fin && finite_bits(yn);
  }
  e2 = gsum(g, e2);
  fin = gall(g, fin);
  g.sync();
  so.err = sqrt(div_rn(e2, (double)m));
  so.good = fine && fin;
  return so;
}

struct IntOpts {
  double rtol, atol, h_init, h_min;
  int max_substeps, max_nonfinite;
  unsigned long long deadline_ns;   // 0: none
  double* trace;                    // optional step trace (see chem_integrate_opts)
  int trace_cap;
  int N;
  // optional tape for the discrete adjoint: accepted step sizes rec_h[i*N + c] (i < rec_cap) and
  // checkpoints rec_ck[(j*m + l)*N + c] = state component l after j*rec_K accepted steps; rec_n[c] is the
  // number of accepted steps, or -1 when the tape overflowed
  double* rec_h;
  double* rec_ck;
  int* rec_n;
  int rec_cap, rec_K;
  int method;   // 0 RODAS3, 1 ROS2, 2 RODAS4
};

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// A cell between two attempts.
struct CellRun {
  int cell = -1;   // -1: none
  bool active = false, rejected_last = false, need_jac = true;
  int nonfinite = 0, ns = 0, na = 0, status = kCellOk;
  double p = 1e5, t = 0.0, dt = 0.0, h = 1.0;
};

// Start the cell whose state sits in y (shared memory); h_io: its proposed first step.
template <class Gs, class MV, class LT>
__device__ __forceinline__ void cell_start(const MV& M, double* sd, const LT& L, int cell, double p, double dt,
                                           double h_io, const IntOpts& o, const Gs& g, CellRun& r) {
  const SPtr y = shared_ptr(sd) + L.y;
  r = CellRun();
  r.cell = cell;
  // input check
  const double T0 = y[0];
  bool ok = isfinite(p) && p > 0.0 && isfinite(dt) && dt >= 0.0 && isfinite(T0) && T0 > 0.0;
  double sig = 0.0;
  for (int k = g.lane; k < M.n; k += g.size) {
    const double yk = y[1 + k];
    ok = ok && isfinite(yk);
    sig = fma(yk, __ldg(M.sp + k), sig);
  }
  sig = gsum(g, sig);
  ok = gall(g, ok) && sig > 0.0;
  r.h = h_io;
  if (!ok) {
    r.status = kCellBadInput;
    if (o.rec_h && g.lane == 0) o.rec_n[cell] = -1;
    return;
  }
  r.p = p;
  r.dt = dt;
  r.h = (h_io > 0.0 && isfinite(h_io)) ? h_io : o.h_init;
  if (dt > 0.0) r.h = fmin(r.h, dt);
  if (o.rec_h)
    for (int i = g.lane; i < M.m; i += g.size) o.rec_ck[(size_t)i * o.N + cell] = y[i];
  r.active = less_pos(r.t, dt);
}

// One attempt of every active cell of the warp (of this group's cell): the groups of a warp stay together.  r.active
// falls when the cell has reached its dt or ends with another status.
template <class Gp, class MV, class LT>
__device__ __forceinline__ void cell_step(const MV& M, double* sd, const LT& L, const IntOpts& o, const Gp& g,
                                          CellRun& r) {
  const SPtr s = shared_ptr(sd), y = s + L.y;
  const int m = M.m;
  bool last = false;
  double hu = r.h;
  if (r.active) {
    last = !less_pos(r.t + r.h, r.dt * (1.0 - 1e-14));
    hu = last ? r.dt - r.t : r.h;
    int st = kCellOk;
    if (r.ns >= o.max_substeps) {
      st = kCellMaxSteps;
    } else if (o.deadline_ns) {
      const auto gs = solo(g);
      const unsigned long long now = (unsigned long long)gbcast(gs, gs.lane == 0 ? (long long)global_ns() : 0ll);
      if (now > o.deadline_ns) st = kCellTimeout;
    }
    if (st == kCellOk && less_pos(hu, o.h_min)) st = kCellHmin;
    if (st != kCellOk) {
      r.status = st;
      r.active = false;
    }
  }
  if (!any_cell(g, r.active)) return;
  const StepOut so = ros_attempt(M, sd, L, r.p, hu, o.rtol, o.atol, g, o.method, any_cell(g, r.active && r.need_jac));
  bool accepted = false;
  if (r.active) {
    ++r.ns;
    r.need_jac = false;
    const bool numbers = so.good && finite_bits(so.err);
    accepted = numbers && leq_pos(so.err, 1.0);
    if (o.trace && g.lane == 0 && r.ns <= o.trace_cap)
      o.trace[(size_t)(r.ns - 1) * o.N + r.cell] = accepted ? hu : -hu;
    if (!numbers) {
      if (++r.nonfinite >= o.max_nonfinite) {
        r.status = kCellNonfinite;
        r.active = false;
      } else {
        r.h = hu * 0.1;
        r.rejected_last = true;
      }
    } else {
      r.nonfinite = 0;
      // step-size factor: err^(-1/(embedded order + 1)): 3 for RODAS3, 2 for ROS2, 4 for RODAS4
      const double fac =
          max_pos(0.2, 0.9 * pow(so.err, o.method == 1 ? -0.5 : o.method == 2 ? -0.25 : -1.0 / 3.0));
      r.h = hu * min_pos(accepted && !r.rejected_last ? 6.0 : 1.0, fac);
      r.rejected_last = !accepted;
      if (accepted) {
        r.t = last ? r.dt : r.t + hu;
        ++r.na;
        r.need_jac = true;
        r.active = less_pos(r.t, r.dt);
        const SPtr yt = s + L.ytmp;
        for (int i = g.lane; i < m; i += g.size) y[i] = yt[i];
      }
    }
  }
  g.sync();
  if (accepted && o.rec_h && r.na <= o.rec_cap) {
    if (g.lane == 0) o.rec_h[(size_t)(r.na - 1) * o.N + r.cell] = hu;
    if (r.na % o.rec_K == 0)
      for (int i = g.lane; i < m; i += g.size) o.rec_ck[((size_t)(r.na / o.rec_K) * m + i) * o.N + r.cell] = y[i];
  }
}

// What is left to record of a cell that has ended.
template <class Gs>
__device__ __forceinline__ void cell_end(const IntOpts& o, const Gs& g, const CellRun& r) {
  if (g.lane != 0) return;
  if (o.trace && r.status != kCellBadInput && r.ns < o.trace_cap) o.trace[(size_t)r.ns * o.N + r.cell] = 0.0;
  if (o.rec_h && r.status != kCellBadInput) o.rec_n[r.cell] = (r.na <= o.rec_cap && r.status == kCellOk) ? r.na : -1;
}

}  // namespace chemgb
