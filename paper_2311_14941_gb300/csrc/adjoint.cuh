// adjoint.cuh -- discrete adjoint of the RODAS3 integration (one warp per cell).
//
// The forward pass records the accepted step sizes and a checkpoint every K accepted steps.  The reverse
// pass walks the segments backwards, recomputes a segment's states from its checkpoint with the same
// arithmetic as the forward pass, and applies the adjoint of each step in reverse order.  Gradients are
// those of the discrete map with the accepted step sizes frozen.
//
// Adjoint of one step (transformed form, M = I/(h gamma) - J(y), A U_i = r_i):
//   mu_i = m_i lambda';  for i = 4..1:  w_i = M^-T mu_i;  mu_j += (c_ij/h) w_i (j < i);
//     stage states Y_i = y + sum_j a_ij U_j:  g_i = J(Y_i)^T w_i,  lambda += g_i,  mu_j += a_ij g_i;
//     Hessian term (J depends on y):           lambda += d/de [J(y + e U_i)^T w_i]
//     parameters theta_j = (ln A_j, Ea_j):     dL/dtheta += w_i^T f_theta(Y_i) + w_i^T J_theta(y) U_i
//   lambda (= dL/dy_n) = lambda' + sum of the above.
// With J = S + u v^T: J^T w = S^T w + v (u.w), and M^-T x by Sherman-Morrison on the transposed factor.
// A shift of ln A_j scales reaction j's forward and reverse rates (both fall-off limits for Troe), so
// d f / d lnA_j = e_j q_j with e_j = d f / d q_j, and d f / d Ea_j = -e_j q_j / (Ru T); w^T e_j is a
// sum over the reaction's participants of a_k = W_k w_k / rho - w_T H_k / (rho c_p).
// The Hessian and the mixed parameter terms use forward-mode dual numbers through the same rate code (exact, no
// finite differences).
#pragma once
#include "device.cuh"

namespace chemgb {

// Memory of the reverse pass.  Shared memory holds the forward cell layout L only (the factor shares
// its region with the Jacobian's pass scratch, as in the integrator), so as many warps per SM fit as
// for the forward pass.  Everything else of a warp lives in its own slice of global memory (offsets in
// doubles below), read and written lane-strided, except the step records (the step's Jacobian and
// factor), which the transposed solves and the products with J(y)^T read by index.
struct AdjLayout {
  CellLayout L;        // shared memory: the forward layout
  CellLayout Ld;       // the dual-number cell of the second-order terms, in dual numbers (contract)
  int dual_bytes;      // its size; in the warp's shared memory, or (dual_shared 0) in its contraction workspace
  int slots;           // contracted derivative slots and the partial sums of their gather
  int dual_shared, slots_shared;   // slots_shared: doubles of them fit the Jacobian's place in the cell
  int ctr;             // contraction workspace, doubles per warp
  int Y3, Y4, W1, W2, W3, W4, MU1, MU2, MU3, MU4, LAM, G, ZT, WS;   // m-vectors
  // step record, kept by the segment recompute for every step of the segment (offsets within a record):
  int SY;              // nnz_S: S at y (the step's own Jacobian)
  int UY, VY;          // m each: the rank-one part u v^T at y
  int HY;              // n: h/RT at y
  int QY;              // R: rates of progress at y
  int SC;              // 8: T, rho, c_p, 1/rho at y
  int LUG;             // nnz_LU + m: the step's factor and its reciprocal pivots
  int JREC, jstride;   // K records of jstride doubles
  int UST;             // K * 4m: U1..U4 of every step of the current segment
  int SEG;             // K * m: the segment's states
  int GA, GE;          // R each: the cell's gradient accumulators (compiled reaction order)
  int total;           // doubles per block
  // sums of the second half of the second-order terms, behind it (m doubles, GA, GE), and their size: apart from the
  // first half's with one warp per cell as with two, so that a cell's gradient does not depend on how many cells a call has
  int GA2, GE2, second;
};

// out = J^T w = S^T w + v (u . w) with S in the internal entry order
template <class P, class Q>
__device__ __forceinline__ void vjp(const MechView& M, P S, P u, P v, const double* w, double* out, Q part,
                                    const Grp1& g) {
  using Sc = double;
  gather_xy(M.g_col, out + 1, part, S, w + 1, g);
  Sc t0 = Sc(0.0), uw = Sc(0.0);
  for (int k = g.lane; k < M.n; k += g.size) t0 = sfma(Sc(S[M.nY + k]), Sc(w[1 + k]), t0);
  for (int i = g.lane; i < M.m; i += g.size) uw = sfma(Sc(u[i]), Sc(w[i]), uw);
  t0 = gsum(g, t0);
  uw = gsum(g, uw);
  for (int c = g.lane; c < M.m; c += g.size) {
    const Sc base = (c == 0) ? t0 : out[c];
    out[c] = sfma(Sc(v[c]), uw, sfma(Sc(S[M.nY + M.n + c]), Sc(w[0]), base));
  }
  g.sync();
}

// sum of a over a reaction's product occurrences minus the sum over its reactant occurrences.
template <class Sc, class P>
__device__ __forceinline__ Sc net_of(const RxRec& r, P a) {
  const int nro = (r.flags >> 1) & 3, npo = (r.flags >> 3) & 3;
  Sc E = a[r.r2p0 >> 16];
  if (npo > 1) E += Sc(a[r.p12 & 0xffff]);
  if (npo > 2) E += Sc(a[r.p12 >> 16]);
  E -= Sc(a[r.r01 & 0xffff]);
  if (nro > 1) E -= Sc(a[r.r01 >> 16]);
  if (nro > 2) E -= Sc(a[r.r2p0 & 0xffff]);
  return E;
}

// dL/dtheta += w^T f_theta at an evaluated state: for reaction r, q_r * E_r with E_r = sum_products a_k -
// sum_reactants a_k, a_k = W_k w_k / rho - w_T H_k / (rho c_p).  hRT, q: the evaluation's h/RT and rates
// of progress; a: n doubles of scratch (shared memory, read by index).
template <class P>
__device__ __forceinline__ void theta_terms(const MechView& M, P hRT, P q, double T,
                                            double rho, double cp, double irho, const double* w, SPtr a,
                                            double* GA, double* GE, const Grp1& g) {
  const double c1 = div_rn((w[0] * kRu) * T, rho * cp);
  for (int k = g.lane; k < M.n; k += g.size)
    a[k] = fma(__ldg(M.sp + M.n + k) * w[1 + k], irho, -(c1 * (double)hRT[k]));
  g.sync();
  const double iRT = rcp_rn(kRu * T);
  for (int r = g.lane; r < M.R; r += g.size) {
    const double E = net_of<double>(ld_rx(M, r).i, a);
    const double qE = q[r] * E;
    GA[r] += qE;
    GE[r] += -(qE * iRT);
  }
  g.sync();
}

// x <- A^-T x (transposed substitution with the factor LU and the reciprocal pivots behind it; x in shared memory)
__device__ __forceinline__ void lu_solveT(const MechView& M, SPtr LU, SPtr x, const Grp1& g) {
  run_fma<false>(M.svT, LU, x, g.lane, g.size, g);
}

// x <- M^-T x with M^T = A^T - v u^T:  x = A^-T x + zt (u . A^-T x) / (1 - u . zt),  zt = A^-T v
__device__ __forceinline__ void smT_solve(const MechView& M, SPtr LU, const double* u, const double* zt, SPtr x,
                                          double idenT, const Grp1& g) {
  lu_solveT(M, LU, x, g);
  double d = 0.0;
  for (int i = g.lane; i < M.m; i += g.size) d = fma(u[i], x[i], d);
  d = gsum(g, d) * idenT;
  for (int i = g.lane; i < M.m; i += g.size) x[i] = fma(zt[i], d, x[i]);
  g.sync();
}

template <class P, class Q>
__device__ __forceinline__ void vset(P dst, Q src, int m, const Grp1& g) {
  for (int i = g.lane; i < m; i += g.size) dst[i] = src[i];
  g.sync();
}

// ---- products with the Jacobian without the Jacobian.  With f_k = W_k w_k / rho, f_T = -sum H_k w_k / (rho c_p) and
// a_k = W_k w_k(weight) / rho - w_T H_k / (rho c_p), the product w^T f is sum_r q_r E_r with E_r = sum_k nu_rk a_k,
// and J^T w is its derivative at fixed weights:
//   through the rates:  G_T = sum_r E_r dq_r/dT,  G_j = sum_r E_r dq_r/dC_j  (at fixed total concentration),
//                       C_j = rho Y_j / W_j:  out_T += G_T - Q/T,  out_j += (rho G_j - Q Wbar) / W_j,  Q = sum_j G_j C_j;
//   through a_k:        out_T += g/T - w_T Ru sum_k w_k cpR_k / (rho c_p) - w_T f_T Ru dcps / c_p,
//                       out_j += (g Wbar - w_T f_T Ru cpR_j / c_p) / W_j,  g = sum_r q_r E_r.
// So a reaction leaves one number per derivative slot, added up by column, where the Jacobian would add it to a row
// for each of its species: at 53 species / 325 reactions 1,436 terms instead of 7,000, and no S, row and column
// sums.  The parameter terms are q_r E_r itself.  In dual numbers the same code gives the derivative of J^T w
// along the tangents: tangent st goes with weight st, and only the tangents of the results are kept.
//
// Tangents carried per dual-number evaluation: the four stages take 4 / kTangentsPerPass passes (fewer live registers
// per dual number against a little more arithmetic per pass).
constexpr int kTangentsPerPass = 2;
using ContractDual = DualN<kTangentsPerPass>;
using ContractVec = DualN<2 * kTangentsPerPass - 1>;   // a number pair (value, tangent) per weight

template <class Sc>
struct Weights;
template <>
struct Weights<double> {   // one weight; results are values
  static constexpr int n = 1;
  using E = double;
  using Vec = double;
  static __device__ __forceinline__ double pick(double x, int) { return x; }
  static __device__ __forceinline__ double get(double v, int) { return v; }
  static __device__ __forceinline__ void set(double& v, int, double e) { v = e; }
  static __device__ __forceinline__ double result(double e) { return e; }
};
template <>
struct Weights<ContractDual> {   // one weight per tangent; results are tangents
  static constexpr int n = kTangentsPerPass;
  using E = Dual;
  using Vec = ContractVec;
  static __device__ __forceinline__ Dual pick(const ContractDual& x, int st) { return Dual(x.v, x.d[st]); }
  static __device__ __forceinline__ Dual get(const ContractVec& v, int st) {
    return st == 0 ? Dual(v.v, v.d[0]) : Dual(v.d[2 * st - 1], v.d[2 * st]);
  }
  static __device__ __forceinline__ void set(ContractVec& v, int st, Dual e) {
    if (st == 0) { v.v = e.v; v.d[0] = e.d; }
    else { v.d[2 * st - 1] = e.v; v.d[2 * st] = e.d; }
  }
  static __device__ __forceinline__ double result(Dual e) { return e.d; }
};

// Takes a reaction's results as eval_reactions produces them.
template <class Sc>
struct ToContraction {
  using W = Weights<Sc>;
  using E = typename W::E;
  using Vec = typename W::Vec;
  const E* a;             // [weights][n]
  const Sc* hRT;
  const Sc* cpR;
  Vec* slots;
  double* GA;
  double* GE;
  int n;
  E iRT[W::n], e[W::n], G_T[W::n], g[W::n];
  Sc sh, scp;             // sum_r q_r times the reaction's change of h/RT and of cp/R
  bool idle = false;      // the reaction changes nothing: its rate, infinite or NaN perhaps, must not count
  __device__ __forceinline__ void rate(int r, const RxRec& rec, const Sc& q) {
    idle = (rec.flags & RXF_IDLE) != 0;
    if (idle) return;
    double dA = 0.0, dE = 0.0;
#pragma unroll
    for (int st = 0; st < W::n; ++st) {
      e[st] = net_of<E>(rec, a + st * n);
      const E qe = W::pick(q, st) * e[st];
      dA += W::result(qe);
      dE += W::result(-(qe * iRT[st]));
      g[st] += qe;
    }
    GA[r] += dA;
    GE[r] += dE;
    sh = sfma(q, net_of<Sc>(rec, hRT), sh);
    scp = sfma(q, net_of<Sc>(rec, cpR), scp);
  }
  __device__ __forceinline__ void dT(int, const Sc& v) {
    if (idle) return;
#pragma unroll
    for (int st = 0; st < W::n; ++st) G_T[st] += e[st] * W::pick(v, st);
  }
  __device__ __forceinline__ void slot(int i, const Sc& v) {
    Vec x;
#pragma unroll
    for (int st = 0; st < W::n; ++st) W::set(x, st, e[st] * W::pick(v, st));
    slots[i] = x;
  }
};

// out (m) = J(y)^T w, or for dual numbers the sum over the weights of the tangents of J(y)^T w_st; GA, GE += the
// parameter terms.  s: the cell (layout L, numbers Sc: y .. cpR, U1 for a, U2 for the column sums); slots: M.n_dslot
// numbers and the partial sums of their gather.
template <class Sc>
__device__ __forceinline__ void contract(const MechView& M, Sc* s, const CellLayout& L, const Sc* y, double p,
                                         const double* const* ws, typename Weights<Sc>::Vec* slots, double* out,
                                         double* GA, double* GE, const Grp1& g) {
  using W = Weights<Sc>;
  using E = typename W::E;
  using Vec = typename W::Vec;
  const ScalT<Sc> sc = eval_species(M, s, L, y, p, g, true);
  E* a = reinterpret_cast<E*>(s + L.U1);
  Vec* col = reinterpret_cast<Vec*>(s + L.U2);
  const Sc* hRT = s + L.hRT;
  const Sc* cpR = s + L.cpR;
  const Sc* C = s + L.C;
  ToContraction<Sc> to{a, hRT, cpR, slots, GA, GE, M.n, {}, {}, {}, {}, Sc(0.0), Sc(0.0)};
#pragma unroll
  for (int st = 0; st < W::n; ++st) {
    const double* w = ws[st];
    const E c1 = sdiv(E((w[0] * kRu) * W::pick(sc.T, st)), E(W::pick(sc.rho, st) * W::pick(sc.cp, st)));
    const E irho = W::pick(sc.irho, st);
    for (int k = g.lane; k < M.n; k += g.size)
      a[st * M.n + k] = sfma(E(__ldg(M.sp + M.n + k) * w[1 + k]), irho, -(c1 * W::pick(hRT[k], st)));
    to.iRT[st] = srcp(E(kRu * W::pick(sc.T, st)));
    to.G_T[st] = E(0.0);
    to.g[st] = E(0.0);
  }
  g.sync();
  eval_reactions<Sc>(M, s, L, sc, g, 0, M.R, true, to);
  {
    auto ld = [&](int i, int) { return slots[i]; };
    auto fin = [](const Vec& v, int) { return v; };
    run_gather<false>(M.g_slot, col, slots + M.n_dslot, ld, fin, g);
  }
  const Sc sh = gsum(g, to.sh), scp = gsum(g, to.scp);
  E gq[W::n], cT[W::n];   // g - Q, and w_T f_T Ru / c_p
  double res_T = 0.0;
#pragma unroll
  for (int st = 0; st < W::n; ++st) {
    E Q = E(0.0);
    for (int j = g.lane; j < M.n; j += g.size) Q = sfma(W::get(col[j], st), W::pick(C[j], st), Q);
    Q = gsum(g, Q);
    const E gt = gsum(g, to.g[st]), GT = gsum(g, to.G_T[st]);
    const E T = W::pick(sc.T, st), cp = W::pick(sc.cp, st), rcp = W::pick(sc.rho, st) * cp;
    const double wR = ws[st][0] * kRu;
    gq[st] = gt - Q;
    const E ircp = srcp(rcp);
    cT[st] = sdiv(E(wR * (-kRu * T * W::pick(sh, st) * ircp)), cp);
    res_T += W::result(GT + gq[st] * W::pick(sc.invT, st) - wR * W::pick(scp, st) * ircp - cT[st] * W::pick(sc.dcps, st));
  }
  for (int j = g.lane; j < M.n; j += g.size) {
    double res = 0.0;
#pragma unroll
    for (int st = 0; st < W::n; ++st)
      res += W::result(sfma(W::pick(sc.rho, st), W::get(col[j], st),
                            gq[st] * W::pick(sc.Wbar, st) - cT[st] * W::pick(cpR[j], st)));
    out[1 + j] = res * __ldg(M.sp + j);
  }
  if (g.lane == 0) out[0] = res_T;
  g.sync();
}

// Second-order terms of kTangentsPerPass stages of one step: J(y)^T W_st differentiated along U_st, the state part into
// out (m), the parameter part into GA, GE.  cell: the dual-number cell (shared memory, which holds nothing else then, or
// global).
__device__ __forceinline__ void second_order_terms(const MechView& M, ContractDual* cell, const CellLayout& Ld,
                                                   ContractVec* slots, const double* y, double p,
                                                   const double* const* Us, const double* const* Ws, double* out,
                                                   double* GA, double* GE, const Grp1& g) {
  ContractDual* yd = cell + Ld.y;
  for (int i = g.lane; i < M.m; i += g.size) {
    ContractDual x(y[i]);
#pragma unroll
    for (int st = 0; st < kTangentsPerPass; ++st) x.d[st] = Us[st][i];
    yd[i] = x;
  }
  g.sync();
  contract<ContractDual>(M, cell, Ld, yd, p, Ws, slots, out, GA, GE, g);
}

// One adjoint step at state y with step h, whose stage vectors U1..U4 and step record jr (the Jacobian
// at y and the factor of the step) the segment recompute kept, up to the second-order terms.  lambda (A.LAM) is
// updated in place, the parameter gradients accumulate into GA, GE; W1..W4 are left in the workspace.
__device__ __forceinline__ void adjoint_stages(const MechView& M, double* s, double* ws, const AdjLayout& A, double* ctr,
                                             const double* jr, const double* y, const double* U1, const double* U2,
                                             const double* U3, const double* U4, double p, double h, double* GA,
                                             double* GE, const Grp1& g) {
  const CellLayout& L = A.L;
  const int m = M.m;
  const double ih = rcp_rn(h);
  double* W1 = ws + A.W1; double* W2 = ws + A.W2; double* W3 = ws + A.W3; double* W4 = ws + A.W4;
  double* MU1 = ws + A.MU1; double* MU2 = ws + A.MU2; double* MU3 = ws + A.MU3; double* MU4 = ws + A.MU4;
  double* LAM = ws + A.LAM; double* G = ws + A.G; double* Y3 = ws + A.Y3; double* Y4 = ws + A.Y4;
  const double* UY = jr + A.UY; const double* VY = jr + A.VY; double* ZT = ws + A.ZT;
  const double* LUg = jr + A.LUG;
  const SPtr X = shared_ptr(s + L.U3);      // shared scratch of the transposed solves
  const SPtr a = shared_ptr(s + L.ytmp);    // shared scratch of the parameter terms (n <= m)
  // ---- the step's factor (kept by the recompute) into shared memory for the first solves
  vset(s + L.LU, LUg, M.nnz_LU + m, g);
  const SPtr LUs = shared_ptr(s + L.LU);
  // transposed Sherman-Morrison vector zt = A^-T v
  vset(X, VY, m, g);
  lu_solveT(M, LUs, X, g);
  double uz = 0.0;
  for (int i = g.lane; i < m; i += g.size) uz = fma(UY[i], X[i], uz);
  uz = gsum(g, uz);
  const double idenT = rcp_rn(1.0 - uz);
  vset(ZT, X, m, g);
  // ---- reverse sweep over the stages, one pass of the loop per stage, so that the kernel holds one copy
  //      of the transposed solve and of the stage Jacobian code (written out, the stages overflowed the
  //      instruction cache)
  for (int i = g.lane; i < m; i += g.size) {
    MU1[i] = M1 * LAM[i]; MU2[i] = 0.0; MU3[i] = M3 * LAM[i]; MU4[i] = M4 * LAM[i];
    Y4[i] = fma(A43, U3[i], fma(A41, U1[i], y[i]));
    Y3[i] = fma(A31, U1[i], y[i]);
  }
  g.sync();
  double* const Wv[4] = {W1, W2, W3, W4};
  double* const MUv[4] = {MU1, MU2, MU3, MU4};
#pragma unroll 1
  for (int st = 3; st >= 0; --st) {   // stage st + 1
    // the factor back into shared memory where a stage Jacobian took its region
    if (st == 2 || st == 1) vset(s + L.LU, LUg, M.nnz_LU + m, g);
    vset(X, MUv[st], m, g);
    smT_solve(M, LUs, UY, ZT, X, idenT, g);
    double* W = Wv[st];
    vset(W, X, m, g);
    if (st >= 2) {
      // stage 4: r4 = f(Y4) + (c41 U1 + c42 U2 + c43 U3)/h, Y4 = y + a41 U1 + a43 U3;
      // stage 3: r3 = f(Y3) + (c31 U1 + c32 U2)/h,          Y3 = y + a31 U1
      const double* w1[1] = {W};
      contract<double>(M, s, L, st == 3 ? Y4 : Y3, p, w1, A.slots_shared ? s + L.S : ctr, G, GA, GE, g);
      if (st == 3) {
        for (int i = g.lane; i < m; i += g.size) {
          MU1[i] = fma(C41 * ih, W4[i], fma(A41, G[i], MU1[i]));
          MU2[i] = fma(C42 * ih, W4[i], MU2[i]);
          MU3[i] = fma(C43 * ih, W4[i], fma(A43, G[i], MU3[i]));
          LAM[i] += G[i];
        }
      } else {
        for (int i = g.lane; i < m; i += g.size) {
          MU1[i] = fma(C31 * ih, W3[i], fma(A31, G[i], MU1[i]));
          MU2[i] = fma(C32 * ih, W3[i], MU2[i]);
          LAM[i] += G[i];
        }
      }
    } else if (st == 1) {   // stage 2: r2 = f(y) + (c21/h) U1 (stage 1: r1 = f(y), nothing to propagate)
      for (int i = g.lane; i < m; i += g.size) MU1[i] = fma(C21 * ih, W2[i], MU1[i]);
    }
    g.sync();
  }
  double* WS = ws + A.WS;
  for (int i = g.lane; i < m; i += g.size) WS[i] = W1[i] + W2[i];
  g.sync();
  vjp(M, jr + A.SY, UY, VY, (const double*)WS, G, shared_ptr(s + L.part), g);
  for (int i = g.lane; i < m; i += g.size) LAM[i] += G[i];
  g.sync();
  theta_terms(M, jr + A.HY, jr + A.QY, jr[A.SC], jr[A.SC + 1], jr[A.SC + 2], jr[A.SC + 3], WS, a, GA, GE, g);
}

// Reverse pass of one cell from its tape.  ws, ctr: the block's global workspaces.  Returns false on a singular factor.
// With two warps, warp 1 takes the second half of each step's second-order terms, which need only the step's state,
// stage vectors and weights: its dual-number cell lies behind the first warp's shared memory, its sums behind the
// first warp's workspace, and it waits at the block's barrier for the rest of the step.  Both warps run one copy of the
// code.  53 species / 325 reactions, igniting cells to 2 us: 308 ms instead of 384 at 300 cells (two fifths of a step
// are these terms), 455-472 instead of 480-490 at 600.
template <int kWarps>
__device__ __forceinline__ bool adjoint_cell(const MechView& M, double* s, double* ws, const AdjLayout& A, double* ctr,
                                             double p, int n_acc, const double* rec_h, const double* rec_ck, int K,
                                             int N, int cell, const Grp1& g, const IntOpts& o, int w) {
  const int m = M.m;
  const CellLayout& L = A.L;
  double* seg = ws + A.SEG;
  double* ust = ws + A.UST;
  double* ws2 = ws + A.total;   // the sums of the second half of the second-order terms
  ContractVec* slots = reinterpret_cast<ContractVec*>(ctr + (size_t)w * A.ctr);
  ContractDual* dual = A.dual_shared ? reinterpret_cast<ContractDual*>(s + (size_t)w * L.total)
                                     : reinterpret_cast<ContractDual*>(slots + A.slots);
  const int nseg = (n_acc + K - 1) / K;
  for (int sg = nseg - 1; sg >= 0; --sg) {
    const int n0 = sg * K, n1 = min(n_acc, n0 + K);
    bool ok = true;
    if (w == 0)
      for (int i = g.lane; i < m; i += g.size) seg[i] = rec_ck[((size_t)sg * m + i) * N + cell];
    g.sync();
    // recompute the segment's states and stage vectors with the forward arithmetic, and keep each step's
    // Jacobian at y and its factor for the reverse sweep
    for (int nn = n0; w == 0 && nn < n1; ++nn) {
      double* jr = ws + A.JREC + (size_t)(nn - n0) * A.jstride;
      vset(s + L.y, seg + (size_t)(nn - n0) * m, m, g);
      auto record = [&](const Scal& sy) {
        vset(jr + A.SY, s + L.S, M.nnz_S, g);
        vset(jr + A.UY, s + L.u, m, g);
        vset(jr + A.VY, s + L.v, m, g);
        vset(jr + A.QY, s + L.q, M.R, g);
        vset(jr + A.HY, s + L.hRT, M.n, g);
        if (g.lane == 0) {
          jr[A.SC] = sy.T; jr[A.SC + 1] = sy.rho; jr[A.SC + 2] = sy.cp; jr[A.SC + 3] = sy.irho;
        }
      };
      const StepOut so = ros_attempt(M, s, L, p, rec_h[(size_t)nn * N + cell], o.rtol, o.atol, g, 0, true, record);
      ok = so.good;   // false also for a singular factor (cannot happen for a step the forward pass accepted)
      if (!ok) break;
      vset(jr + A.LUG, s + L.LU, M.nnz_LU + m, g);
      double* u4 = ust + (size_t)(nn - n0) * 4 * m;
      for (int i = g.lane; i < m; i += g.size) {
        u4[i] = s[L.U1 + i]; u4[m + i] = s[L.U2 + i]; u4[2 * m + i] = s[L.U3 + i]; u4[3 * m + i] = s[L.U4 + i];
        if (nn + 1 < n1) seg[(size_t)(nn - n0 + 1) * m + i] = s[L.ytmp + i];
      }
      g.sync();
    }
    if (kWarps > 1) ok = __syncthreads_and(ok);
    if (!ok) return false;
    for (int nn = n1 - 1; nn >= n0; --nn) {
      const double* u4 = ust + (size_t)(nn - n0) * 4 * m;
      const double* y = seg + (size_t)(nn - n0) * m;
      double* LAM = ws + A.LAM;
      if (w == 0)
        adjoint_stages(M, s, ws, A, ctr, ws + A.JREC + (size_t)(nn - n0) * A.jstride, y, u4, u4 + m, u4 + 2 * m,
                       u4 + 3 * m, p, rec_h[(size_t)nn * N + cell], ws + A.GA, ws + A.GE, g);
      if (kWarps > 1) __syncthreads();
      // Hessian and mixed parameter terms: J(y)^T w_i differentiated along U_i, kTangentsPerPass stages at a time
      const double* Us[4] = {u4, u4 + m, u4 + 2 * m, u4 + 3 * m};
      const double* Ws[4] = {ws + A.W1, ws + A.W2, ws + A.W3, ws + A.W4};
#pragma unroll 1
      for (int s0 = w * kTangentsPerPass; s0 < 4; s0 += kWarps * kTangentsPerPass) {
        double* G = s0 == 0 ? ws + A.G : ws2;
        second_order_terms(M, dual, A.Ld, slots, y, p, Us + s0, Ws + s0, G, s0 == 0 ? ws + A.GA : ws2 + A.GA2,
                           s0 == 0 ? ws + A.GE : ws2 + A.GE2, g);
        if (kWarps > 1) __syncthreads();
        if (w == 0)
          for (int i = g.lane; i < m; i += g.size) {
            LAM[i] += G[i];
            if (kWarps > 1) LAM[i] += ws2[i];
          }
        g.sync();
      }
    }
  }
  return true;
}

}  // namespace chemgb
