// mech.h -- layout of a compiled mechanism, shared by the host compiler and the device kernels.
//
// All tables live in one device allocation; MechView carries typed pointers into it and is passed to
// kernels by value.  Index fields of the warp programs are 16 bits wide, which bounds reactions,
// derivative slots and factor entries to 65535 (chem_create reports CHEM_EUNSUPPORTED beyond).
#pragma once
#ifdef __CUDACC_RTC__
// run-time compilation (mechanism-specialised kernels) has no C library headers
typedef unsigned char uint8_t;
typedef unsigned short uint16_t;
typedef unsigned int uint32_t;
typedef long long int64_t;
typedef unsigned long long uint64_t;
#else
#include <cstdint>
#endif

namespace chemgb {

// Per-cell status codes of the device code (the same values as chem.h's CHEM_CELL_*, checked there).
enum : int { kCellOk = 0, kCellMaxSteps = 1, kCellHmin = 2, kCellNonfinite = 3, kCellBadInput = 4, kCellTimeout = 5 };

constexpr double kRu = 8.314462618;   // J/(mol K)
constexpr double kP0 = 101325.0;      // Pa, standard state of Kc
constexpr int kWarp = 32;
constexpr int kMaxWarpsPerCell = 2;   // a cell is integrated by one warp or by two
// Lane groups that integrate one cell, and the width their warp programs are built for:
//   group 0: one warp (32 lanes), group 1: two warps of a block (64 lanes), group 2: half a warp
//   (16 lanes; two cells share a warp, for mechanisms with few species).
constexpr int kNumGroups = 3;
// Kernels with helper warps, numbered after the lane groups whose programs they run: kHelpWarps[i] helpers for a cell of
// group kHelpGroups[i], those of a group with rising numbers of helpers.
constexpr int kHelpForms = 3;
constexpr int kHelpGroups[kHelpForms] = {0, 0, 1};
constexpr int kHelpWarps[kHelpForms] = {1, 3, 2};
constexpr int kGroupWidth[kNumGroups] = {32, 64, 16};

// ---- species table, structure of arrays: field f of species k at sp[f * n + k], SP_STRIDE fields (lanes hold
// consecutive species, so a warp's read of one field is one or two cache lines instead of 32)
//   [0] 1/W  [1] W  [2] T_mid  [3] unused
//   [4 .. 4+RANGE)   low range, [4+RANGE .. 4+2 RANGE) high range, each:
//   a0 a1 a2 a3 a4 | h1..h4 = a1/2 a2/3 a3/4 a4/5 | g1..g4 = -a1/2 -a2/6 -a3/12 -a4/20 | a5 a6 |
//   d2 d3 d4 = 2a2 3a3 4a4
// so cp/R = a0 + T(a1 + T(a2 + T(a3 + T a4))), h/RT = a0 + T(h1 + ...) + a5/T,
// g = h/RT - s/R = a0 (1 - ln T) + T(g1 + T(g2 + T(g3 + T g4))) + a5/T - a6,
// d(cp/R)/dT = a1 + T(d2 + T(d3 + T d4)).
constexpr int SP_RANGE = 18;
constexpr int SP_STRIDE = 4 + 2 * SP_RANGE;

// ---- reaction tables.  Reactions are ordered Troe, third-body, elementary; within a class and a Jacobian
// pass the simple ones (see RXF_SIMPLE) stand together, so that whole rounds of lanes are simple.
// doubles, structure of arrays (field f of reaction r at rxd[f * R + r]), RX_D fields:
//   [0] ln A  [1] b  [2] Ea/Ru  [3] ln A0  [4] b0  [5] Ea0/Ru  [6] 1-alpha  [7] alpha  [8] 1/T3  [9] 1/T1
//   [10] T2 (0: absent)  [11] unused
constexpr int RX_D = 12;
// ints, RX_I per reaction:
//   [0] type (0 elementary, 1 third-body, 2 Troe)  [1] reversible  [2] reactant occurrences (1..3)
//   [3] product occurrences (1..3)  [4..6] reactant species per occurrence (coefficient nu expands into
//   nu occurrences)  [7..9] product occurrences  [10] sum of net coefficients  [11] efficiency offset
//   [12] efficiency count  [13] derivative-slot offset  [14] derivative-slot count  [15] efficiency offset again
//   ([12..15] are read as one 16-byte word)
constexpr int RX_I = 16;
// one 16-byte record per reaction with what the rate of progress needs: six 16-bit species indices (reactant,
// then product occurrences; absent ones are 0) and the flags below
struct alignas(16) RxRec {
  uint32_t r01, r2p0, p12, flags;   // r0 | r1 << 16, r2 | p0 << 16, p1 | p2 << 16
};
// a listed efficiency (species and efficiency - 1), and a derivative slot: its species' (efficiency - 1), 0 if not
// listed, and the occurrences that are this species (bits 0..2 reactants, 3..5 products)
struct alignas(16) EffRec {
  double am1;
  int sp, pad;
};
struct alignas(16) SlotRec {
  double am1;
  int mask, pad;
};
// flags (bits 16-31: derivative-slot offset): bit 0 reversible, bits 1-2 reactant occurrences, bits 3-4 product occurrences, bit 5 simple
// (elementary, reversible, two reactants and two products, all four different species), bit 6 idle (the same species on
// both sides: no net change)
enum : int { RXF_REV = 1, RXF_SIMPLE = 32, RXF_IDLE = 64 };

// ---- warp programs, compiled for a group of `width` lanes (one warp per cell: 32, two: 64, half: 16)
// The device reads every program in blocks of kProgBlock steps, a block ahead.
constexpr int kProgBlock = 8;
// Gather ("flattened segmented reduction"): step s, lane l executes op[s*width + l]:
//   acc = fma(value(a, b), acc); if dst != NONE: out[dst] = acc, acc = 0.  Padded to whole blocks of steps.
// dst >= PARTIAL_BIT selects the partial-sum buffer; a combine list then adds partials into outputs.
struct GatherOp {
  uint16_t a, b, dst, flags;
};
// flags: padding (no accumulation); in every lane's op of a step in which some lane ends a piece
enum : int { GF_IDLE = 1, GF_END = 2 };
constexpr uint16_t DST_NONE = 0xFFFF;
constexpr uint16_t PARTIAL_BIT = 0x8000;

// Elimination / solve program: step s has one kind; lane l executes op[s*width + l] (t == OP_IDLE: idle).
//   LU:    K_RECIP  dinv[t] = 1 / LU[a]      K_SCALE  LU[t] *= dinv[a]     K_UPDATE LU[t] -= LU[a] * LU[b]
//   solve: K_SCALE  x[t] *= dinv[a]          K_UPDATE x[t] -= LU[a] * x[b]
// Every op of a step, idle ones included, carries the step's kind.
struct ElimOp {
  uint16_t t, a, b, kind;
};
constexpr uint16_t OP_IDLE = 0xFFFF;
enum : int { K_RECIP = 0, K_SCALE = 1, K_UPDATE = 2 };

// The same programs as the device runs them.  v = the factor's entries followed by the negated reciprocals of its
// pivots for the elimination, the right-hand side for a substitution (whose factor is A, as above); an op is
//   v[t] = fma(-A[a], v[b], FM_MUL ? -0 : v[t]),
// an update or (b = t, a = a negated reciprocal) a scaling: fma(x, y, -0) is x y rounded, signed zeros included.
// One form for both needs no branch in a step and lets them share a step.  Updates of one target keep the order
// of the program above, so the results are its results.  A block is up to kProgBlock steps, right-aligned, then
// in the elimination at most one step of reciprocals, v[t] = -1/v[a], in slot kProgBlock.
struct FmaOp {
  uint16_t t, a, b, flags;
};
enum : int { FM_MUL = 1, FM_IDLE = 2 };
struct FmaProgram {
  const FmaOp* ops;   // [blocks * (kProgBlock + recip) * width]
  const int* head;    // [blocks] steps of the block, + 256 with a step of reciprocals
  int blocks;
};

struct Gather {
  const GatherOp* ops;   // [blocks * kProgBlock * width]
  int blocks;
  int n_partial;
  const int* comb;       // [n_comb * 3]: dst, first partial, count
  int n_comb;
};

// The Jacobian's reaction loop runs in passes over consecutive reaction ranges so that a pass's
// dq/dT values and derivative slots fit in the region the LU factor occupies during a step.
constexpr int kMaxJPass = 8;
enum : int { JP_RB = 0, JP_RE = 1, JP_SB = 2, JP_CNT = 3 };   // first/end reaction, first slot, reactions

struct MechView {
  static constexpr int kHelpers = 0;   // helper warps of a cell (HelpedView: kernels that have some)
  int width;                 // lanes of the programs below: the lane group's width (32, 64 or 16)
  int n, R, m;
  int n_troe, n_tb;          // reactions [0, n_troe) Troe, [n_troe, n_troe + n_tb) third-body
  int nY;                    // Y-block entries of S (row-major by species, diagonal included)
  int nnz_S;                 // nY + n (T column) + m (T row)
  int nnz_LU;
  int n_dslot;
  const double* sp;          // [SP_STRIDE * n]
  const double* rxd;         // [RX_D * R]
  const int* rxi;            // [R * RX_I]
  const RxRec* rxr;          // [R]
  const EffRec* eff;         // listed efficiencies
  const SlotRec* dslot;      // [n_dslot]
  const int* entry_row;      // [nY] species k of Y-block entry
  const int* entry_col;      // [nY] species j
  const double* entry_wratio;// [nY] W_k / W_j
  Gather g_omega;            // species <- reactions (a = reaction, b = top 16 bits of double(nu))
  int n_jpass;               // Jacobian passes
  int jpass[kMaxJPass][4];   // per pass: JP_RB, JP_RE, JP_SB, JP_CNT
  Gather g_jac[kMaxJPass];   // per pass: S[0 .. nY + n) += nu * region[a] (a < cnt: dq/dT of reaction
                             // rb + a into the T column; a >= cnt: derivative slot sb + a - cnt into the
                             // Y block), b = top 16 bits of double(nu)
  Gather g_row;              // species k <- sum_j Dtil_kj C_j (a = entry, b = species j)
  Gather g_col;              // species i <- sum_k h_k Dtil_ki (a = entry, b = species k)
  Gather g_slot;             // species j <- derivative slots of column j (one warp per cell only: the adjoint)
  const int* lu_src;         // [nnz_LU] S index feeding the slot (-1: fill)
  const int* lu_diag;        // [m] LU slot of the diagonal of state index s (natural order)
  FmaProgram lu;             // elimination
  FmaProgram sv;             // forward + backward substitution, vector indices in state order
  FmaProgram sv2;            // the same for half of the group's lanes (two right-hand sides at once)
  FmaProgram svT;            // transposed substitution (A^T x = b)
  const int* rx_order;       // [R] compiled reaction -> description index
  const int* s_out;          // [nnz_S] position of internal S entry in the CSR output order
  // tabulated temperature functions (an opt-in approximation; tab_on == 0: every function exact):
  // class c (0 exp(g_k), 1 exp(-g_k), 2 forward rate coefficient, 3 Troe centre) at interval j, function f
  // has its deg[c] + 1 polynomial coefficients (powers of tau) at tab[c] + (j * nfun_c + f) * (deg[c] + 1)
  int tab_on;
  int tab_deg[4];            // 0: the class stays exact
  const double* tab[4];
  double tab_ulo, tab_du;    // interval j covers u = 1/T in [tab_ulo + j du, tab_ulo + (j + 1) du)
  double tab_tlo, tab_thi;   // tabulated range of T
  int tab_ni;                // intervals
};

// The same tables for the kernels whose cells have H helper warps.
template <int H>
struct HelpedView : MechView {
  static constexpr int kHelpers = H;
};

// Per-cell shared-memory layout (offsets in doubles).
struct CellLayout {
  int y, ytmp, f0, U1, U2, U3, U4, x, z, u, v;   // m-vectors
  int C, hRT, eg, emg, cpR;                       // n-vectors
  int q;                                          // R-vector
  int S;                                          // nnz_S
  int LU, dinv;                                   // nnz_LU, m
  int D;                                          // Jacobian pass region (aliases LU and dinv)
  int part;                                       // partial sums of the gathers
  int misc;                                       // 16 scalars
  int total;                                      // doubles per cell
};

}  // namespace chemgb
