// internal.h -- data structures shared by the mechanism compiler (host) and the
// solve kernels (device).  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "chemgpu.h"

namespace chemgpu {

constexpr int QMAX = 5;             // highest BDF order
constexpr int NROW = QMAX + 3;      // history rows D_0 .. D_{QMAX+2}
constexpr int GRID_IMIN = -26;      // step-factor grid g_i = 2^(i/8)
constexpr int GRID_IMAX = 26;
constexpr int GRID_N = GRID_IMAX - GRID_IMIN + 1;
constexpr int WARP = 32;
constexpr int MAX_WARPS_PER_BLOCK = 12;  // cells per block (history and vectors live in registers)
constexpr int ADJ_WARPS_PER_BLOCK = 12;  // most cells per block of the adjoint walk
constexpr int TAN_WARPS_PER_BLOCK = 4;   // ... and of the tangent walk (a larger launch bound costs it
                                         // registers and 70% more instructions)

// A warp program is a sequence of passes of exactly 32 op slots; lane l runs
// slot l of every pass and the warp synchronises between passes.  The
// scheduler guarantees that no location written in a pass is read or written
// by another op of the same pass, so the passes run without intra-pass races.
// On the host an op holds element indices:
//   FMA op:    W[t] = fma(W[a], W[b], W[c])
//   RECIP op:  W[t & 0x7fff] = -1 / W[a]         (t has bit 15 set)
//   empty:     t == 0xffff
// On the device the same op holds BYTE offsets into the cell's work array,
// empty slots become a harmless FMA into a dummy slot, and a RECIP op carries
// c == 0xffff.  A pass with reciprocals may hold FMA ops in its other lanes.
struct Op {
  uint16_t t, a, b, c;
};
constexpr uint16_t OP_EMPTY = 0xffff;
constexpr uint16_t OP_RECIP = 0x8000;
constexpr uint16_t DEV_RECIP = 0xffff;     // device marker in .w of RECIP passes

// Tables read by every warp of every cell, packed into one 16-byte-aligned
// blob per LU precision so that a block can stage them into shared memory
// with one bulk copy.  Byte offsets of each section within the blob:
struct TableOffsets {
  int f_ops, fwd_ops, bwd_ops;     // ushort4 programs (f on Wd, fwd/bwd on WL)
  int f_runs;                      // uint32 run table of the f program
  int rx_slots;                    // uint2 [R]: byte offsets into Wd of the reactants' y
  int pair_rx;                     // int [n_pairs]
  int pair_other;                  // uint32 [n_pairs]: two 16-bit byte offsets into Wd
  int lu_diag;                     // int [S]: byte offsets into WL of the pivot diagonal
  int dconst_off, dconst_val;      // int [d_nconst] byte offsets into Wd, double values
  int Lconst_off, Lconst_val;      // int [L_nconst] byte offsets into WL, double values
  int thr2, thr3, g;               // step-factor grid: thresholds of the raw squared-norm sums
                                   // (biases 2 and 3), double [7][GRID_N] each, and the factors
                                   // g_i, [GRID_N]
  int lim;                         // double [2][8]: by order q, the raw-sum bounds of the error
                                   // test, S (q+1)^2, and of the corrector, S (0.1 (q+1))^2
  int staged;                      // bytes of the prefix the persistent driver stages in shared
                                   // memory (programs and slots used every Newton iteration or
                                   // refactorisation; constants and the grid stay in global memory)
  int bytes;                       // total, a multiple of 16
};

constexpr int RX_EXT = 8;   // extra rate parameters per reaction

// Terms of the tile derivative (MechDev::tl_term): coefficient +1, -1, another
constexpr uint32_t TILE_PLUS = 0, TILE_MINUS = 1, TILE_GENERAL = 2;
constexpr int TILE_CHUNK = 8;     // terms per chunk: the f program's
constexpr int TILE_WARPS = 12;    // warps per group of the tile derivative
constexpr int TILE_GROUPS = 2;    // groups per block

// Everything a solve kernel needs about a mechanism; passed by value.
struct MechDev {
  int S, R, max_reac, n_phot, n_pairs;
  // rate constants (read once per cell)
  const int *rx_kind;      // [R]
  const int *rx_nreac;     // [R]
  const int *rx_phot;      // [R] index among photolysis reactions, or -1
  const double *rx_A, *rx_Ea, *rx_B, *rx_J;
  const double *rx_ext;    // [R][RX_EXT]: A2, Ea2, B2, A3, Ea3, B3, Fc, N (pressure-dependent kinds)
  // reaction data for the derivative-design comparison (chem_eval_deriv_design):
  // the caller's records as uploaded (array of structures), and the same as
  // structure of arrays: reactants [R][3], product counts [R], products and yields [R][8]
  const chem_reaction *rx_aos;
  const int *rx_reac, *rx_nprod, *rx_prod;
  const double *rx_yld;
  // f for tiles of 32 cells, one lane per cell (deriv_gather_kernel): the
  // reactions by their number of reactants; per species the terms of its sum in
  // the f program's order (reaction | TILE_* << 16) with their coefficients; the
  // species dealt to the block's warps
  const uint2 *tl_rx;      // [R] reactions with 1, then 2, then 3 reactants: j | r0 << 16, r1 | r2 << 16
  int tl_rx_end[3];        // ends of those three ranges
  const uint32_t *tl_term; // (two words past the last term are readable)
  const double *tl_nu;     // read for TILE_GENERAL terms
  const int *tl_ptr;       // [S + 1] first term of each species
  const int *tl_list;      // [S] species, warp by warp
  const int *tl_warp;      // [TILE_WARPS + 1] first entry of each warp in tl_list
  int tl_cost, ga_cost;    // FP64 warp instructions per tile, and per cell by the f program
  // species permutation: position of species s in the pivot order
  const int *sp_pos;       // [S]
  // per-cell double array Wd (element indices)
  int Wd_len, d_Y, d_KT, d_RT, d_F, d_ONE, d_ZERO, d_DUMMY;
  // per-cell LU-precision array WL (element indices)
  int WL_len, L_LU, L_X, L_P, L_ZERO, L_DUMMY, nnz_lu;
  int d_nconst, L_nconst;
  int m_clear;             // WL entries [0, m_clear) are cleared before forming M
  int fwd_npass, bwd_npass;
  int f_nruns, m_nruns, lu_nruns;  // run tables (f: in the staged blob; M, LU: m_runs, lu_runs)
  const uint32_t *m_runs, *lu_runs;
  // staged tables: blob[0] for an FP64 LU, blob[1] for an FP32 LU (global memory)
  const unsigned char *blob[2];
  TableOffsets tab;
  // programs streamed from global memory, per LU precision (byte-offset ops)
  const ushort4 *m_ops[2], *lu_ops[2];
  // history rescale T(eta)_{im} = sum_p coef[(i-1)*QMAX + m-1][p] eta^p,
  // i, m = 1..QMAX, p = 0..QMAX
  const double *rescale_coef;
  // ---- discrete adjoint (FP64): after the forward's Wd and WL, mu[S], nm[R] =
  // nu_j . mu, jtm[S] = J^T mu, g[R] (theta gradient), temps, constants (up to
  // Wda_len), then pp[n_pairs] = dr_j/dy_l at a_PP; indices from the start of Wd
  int Wda_len, a_MU, a_NM, a_PP, a_JTM, a_G;
  int a_nconst;
  const int *a_const_off;          // byte offsets into the extended Wd
  const double *a_const_val;
  const ushort4 *nudot_ops, *jt_ops;    // programs on the extended Wd
  const ushort4 *fwdT_ops, *bwdT_ops;   // U^T and L^T solves on WL (FP64 byte offsets)
  int fwdT_npass, bwdT_npass;
  const uint32_t *nudot_runs, *jt_runs;   // run tables of nudot and jt
  int nudot_nruns, jt_nruns;
};

// On the device a program is a sequence of groups of two passes, lane by lane:
// 32 x (op of the first pass, op of the second), so one 16-byte load brings a
// lane's ops of both.  Its run table holds one uint32 per run of equal groups
// (kind << 28 | groups):
//   RUN_PIPE   groups of passes none of which touches what the one before it
//              writes: each pass's operands are loaded while the FMAs of the one
//              before are in flight
//   RUN_PIPE1  the same, the last group with one pass (the second slot not used)
//   RUN_SEQ    groups of two passes, the second after the first
//   RUN_RECIP  two groups, three passes, reciprocals in the first: a lane with a
//              reciprocal spends three FP64 instructions on it and has no op in the
//              other two, every other lane runs its three FMA ops; all ops of the
//              unit are independent of each other
// A program without runs (the triangular solves) is its passes in order.
constexpr uint32_t RUN_PIPE = 0, RUN_PIPE1 = 1, RUN_RECIP = 2, RUN_SEQ = 3;
constexpr int GROUP_BYTES = 2 * WARP * 8;
constexpr int PAD_GROUPS = 5;     // readable groups past a program's last (the interpreters read ahead unconditionally)

struct HostProgram {
  std::vector<Op> ops;   // n_pass * 32
  // per pass: 3 the first pass of a reciprocal unit (the two passes after it,
  // marked 0, belong to it), 0 otherwise
  std::vector<uint8_t> unit;
  // per pass: 1 the first pass of a run, 2 a pass that continues it (it touches
  // nothing the pass before it writes), 0 a pass outside runs
  std::vector<uint8_t> run;
  int n_ops = 0;
  int n_pass() const { return (int)(ops.size() / WARP); }
  // the device form's groups: the passes in each (-1: none), and the run table
  void groups(std::vector<std::pair<int, int>> &g, std::vector<uint32_t> &runs) const {
    for (int p = 0; p < (int)unit.size();) {
      if (unit[p] == 3) {
        if (!runs.empty() && runs.back() >> 28 == RUN_RECIP) runs.back()++;      // units of two groups
        else runs.push_back(RUN_RECIP << 28 | 1u);
        g.push_back({p, p + 1});
        g.push_back({p + 2, -1});
        p += 3;
        continue;
      }
      // [p, e): a run; or passes that each start one (outside runs: the rest)
      auto starts = [&](int x) { return x < (int)unit.size() && unit[x] != 3 && run[x] != 2; };
      int e = p + 1;
      const bool alone = !(e < (int)unit.size() && run[e] == 2);
      if (alone)
        while (starts(e) && !(e + 1 < (int)unit.size() && run[e + 1] == 2)) ++e;
      else
        while (e < (int)unit.size() && run[e] == 2) ++e;
      const uint32_t n = (uint32_t)(e - p);
      if (!alone) {
        runs.push_back((n & 1 ? RUN_PIPE1 : RUN_PIPE) << 28 | (n + 1) / 2);
      } else {
        if (n > 1) runs.push_back(RUN_SEQ << 28 | n / 2);
        if (n & 1) runs.push_back(RUN_PIPE1 << 28 | 1u);
      }
      for (; p < e; p += 2) g.push_back({p, p + 1 < e ? p + 1 : -1});
      p = e;
    }
    runs.push_back(0u);        // the interpreter reads an entry ahead
  }
};

// Compiled mechanism (host + device copies).
struct Mechanism {
  int S = 0, R = 0, n_phot = 0, max_reac = 0, n_pairs = 0, nnz_jac = 0, nnz_lu = 0;
  std::vector<int> pos;              // pivot position of each species
  std::vector<uint8_t> fill;         // S*S in pivot order
  HostProgram f_prog, m_prog, lu_prog, fwd_prog, bwd_prog;
  HostProgram nudot_prog, jt_prog, fwdT_prog, bwdT_prog;   // adjoint
  std::vector<double> a_consts_v;
  std::vector<int> a_consts_i;
  double flops_f = 0, flops_jac = 0, flops_lu = 0, flops_solve = 0;
  double flops_adj_iter = 0, flops_tan_iter = 0;   // per corrector iteration of the adjoint / tangent walks
  // host copies of the small tables that upload_mechanism() sends to the device
  std::vector<double> d_consts_v, L_consts_v;
  std::vector<int> d_consts_i, L_consts_i;
  std::vector<int> pair_rx;
  std::vector<std::pair<int, int>> pair_other;   // Wd element indices
  std::vector<int> lu_diag;                      // WL element indices
  std::vector<int> rx_slot_idx;                  // [R][3] Wd element indices of the reactants' y
  std::vector<std::vector<std::pair<double, int>>> f_terms;   // f_i = sum nu_ij r_j: (nu, j) in the f program's order
  std::vector<chem_reaction> rx;
  MechDev dev{};                     // device pointers filled in upload()
  std::vector<void *> allocations;   // device buffers owned
  int device = 0;
};

// Build the mechanism tables (host).  Returns 0 or a CHEM_E* code with msg.
int compile_mechanism(int S, int R, const chem_reaction *rx, Mechanism &m, std::string &msg);
int upload_mechanism(Mechanism &m, std::string &msg);
void free_mechanism(Mechanism &m);

// Launch the solve kernel for all cells (device side in kernels.cu).
struct CellsDev {
  int64_t n_cells;
  const double *T, *P, *J;      // J may be null (mechanism J)
  const double *theta;          // may be null
  double *y;                    // [S][C] in/out
  chem_cell_stats *stats;       // [C]
  unsigned long long *queue;    // persistent driver work counter (may be null)
  const int *order;             // persistent driver: the queue hands out order[0], order[1], ...;
                                // adjoint / tangent: warp slot i takes cell order[i] (NULL: cell i)
                                // (null: cell index order)
  // staging counters (may be null): [0] blocks whose bulk copy of the tables
  // was not seen to land within the first bounded wait (they read the tables
  // from global memory instead), [1] blocks that exited before seeing that
  // late copy land within the final bounded wait
  unsigned long long *stage;
  // adjoint tape (tape_n null: not recording).  Per cell e < tape_cap events,
  // kq = kind | q << 8, val:
  //   0 INIT      val h0,   row y at the start of the solve
  //   1 RESCALE   q order,  val eta
  //   2 STEP      q order,  val c = h/gamma_q (accepted step)
  //   3 PROJECT   q species projected onto y = 0 by the next STEP
  //   4 REFACTOR  q its row index, val c_M; row y_J (M = I - c_M J(y_J))
  //   5 ITER      q iteration k of the next STEP; row y_k, the iterate it
  //               evaluated f at
  // Rows are numbered in event order over the INIT, REFACTOR and ITER events.
  int *tape_kq;
  double *tape_val;
  double *ytape;                // [C][row_cap][S] rows
  int *tape_n;                  // [C] events so far (kept across solve_step calls)
  int *tape_bad;                // [C] nonzero: overflow or a failed solve, no sensitivity
  int *tape_rows;               // [C] rows so far
  int tape_cap, row_cap;
};

enum TapeKind { EV_INIT = 0, EV_RESCALE = 1, EV_STEP = 2, EV_PROJECT = 3, EV_REFACTOR = 4, EV_ITER = 5 };

// Buffers of chem_sensitivity (device, owned by the batch).
struct AdjDev {
  const double *dLdy;           // [S][C]
  double *dLdy0;                // [S][C]
  double *gcell;                // [R][C] per-cell theta gradients
  double *dLdtheta;             // [R]
  int accumulate;               // 0: dLdtheta = the sum over cells; 1: dLdtheta += that sum
};

// Buffers of chem_tangent (device, owned by the batch).
struct TanDev {
  const double *dy0;            // [S][C] direction in the initial state
  const double *dtheta;         // [R] direction in theta (shared by all cells)
  double *dy;                   // [S][C] out: the directional derivative of the state
};

// Iterations of the bounded wait for a block's bulk copy of the tables.
constexpr long long STAGE_WAIT_DEFAULT = 1LL << 22;

struct LaunchCfg {
  int lu_precision;     // 64 / 32
  int driver;           // CHEM_DRIVER_*
  int regs;             // solve_registers of the batch (a pipeline's chunk: of all its cells)
  int couple;           // > 1: cells integrated in coupled groups of this many (one block each)
  int warps_per_block;
  int blocks_per_sm;
  double rtol, atol, dt;
  int max_order, max_steps;
  int n_steps;          // > 1: that many consecutive steps per cell in one launch (not coupled)
  long long stage_wait; // iterations of the first wait for the staged tables (chem_opts.stage_wait)
};

size_t smem_per_cell(const MechDev &m, int lu_precision);
size_t staged_bytes(const MechDev &m, int driver);   // tables staged per block by the driver
cudaError_t set_constants();   // gamma_m, 1/gamma_m into constant memory of the current device
cudaError_t launch_solve(const MechDev &m, const CellsDev &c, const LaunchCfg &cfg, cudaStream_t stream);
// Cells most expensive first for the persistent queue: per cell its cost in
// the batch's previous solve, or for a first solve the sum of its rate
// constants, bucketed linearly in log2 over the batch's range, then a counting
// sort into order[n_cells].  bucket[n_cells] and hist[ORDER_HIST_INTS] are
// scratch.  Stream-ordered (capturable).
constexpr int ORDER_BUCKETS = 256;
constexpr int ORDER_HIST_INTS = 2 * ORDER_BUCKETS + 2;   // counts, cursors, key range
// The same counting sort keyed by tape length (events), longest first: the
// order in which the adjoint and tangent kernels take the cells.
cudaError_t launch_order_tape(const CellsDev &c, int *bucket, int *hist, int *order, cudaStream_t stream);
// ... and keyed by the cost of coupled groups of G cells: order[i] is a group index.
cudaError_t launch_order_groups(const CellsDev &c, int G, int *bucket, int *hist, int *order, cudaStream_t stream);
// solved: the batch has been solved before, so (nearly) every cell has a cost.
cudaError_t launch_order(const MechDev &m, const CellsDev &c, double rtol, double atol, bool solved, int *bucket, int *hist,
                         int *order, cudaStream_t stream);
int max_warps_per_block(const MechDev &m, int lu_precision, int driver);
// resident blocks per SM of the solve kernel for a block of warps_per_block cells
int occupancy(const MechDev &m, int lu_precision, int driver, int regs, int warps_per_block);
// Registers of a solve kernel's thread.  A sub-partition's 16,384 hold 3 warps at up
// to 168 (a block of 12 warps on the SM), 4 at 128, 6 at 80.  Shared memory holds 12
// cells or fewer of 72 species and more, so those kernels take 168.  Of up to 32
// species it holds 24 and more (ms of a first solve, 20/40, at 168 / 128 / 80):
//   plain driver, more than 12 cells per SM: 128 (FP64: 2,000 cells 2.6 / 2.5 / 2.7,
//   20,000 13.8 / 13.3 / 12.7, 50,000 32.5 / 31.3 / 29.2; but 10 cells at rtol 1e-8
//   3.55 / 3.59 / 4.10, which is why fewer keep 168);
//   FP32 factorisation, more than 80 cells per SM: 80, since what a warp waits for is
//   latency, not the FP64 unit (plain: 5,000 cells 4.0 / 3.7 / 3.7, 10,000 6.8 / 6.0 /
//   5.9, 20,000 12.7 / 11.0 / 10.3, 50,000 29.9 / 25.6 / 23.6; persistent: 2,000 cells
//   2.0 / 2.0 / 2.3, 10,000 5.9 / 5.6 / 5.3 and repeated 4.8 / 4.4 / 4.5, with 32/80
//   6.9 / 7.7 / 8.5, 14,000 7.9 / 7.3 / 6.8, 50,000 25.3 / 23.5 / 21.6);
//   the persistent FP64 kernel 168: its narrow batches gain more from few warps
//   (repeated solve: 3,500 cells 2.7 / 3.3 / 3.3, 20,000 11.3 / 10.9 / 10.8).
inline int register_rule(int n_species, int lu_precision, int driver, int couple, int64_t n_cells, int n_sm) {
  if (n_species > WARP || couple > 1) return 168;
  if (lu_precision == 32 && n_cells > (int64_t)80 * n_sm) return 80;
  if (driver == CHEM_DRIVER_PLAIN && n_cells > (int64_t)12 * n_sm) return 128;
  return 168;
}
int solve_registers(const MechDev &m, int lu_precision, int driver, int couple, int64_t n_cells);
// cells per block that maximises resident cells per SM (0 if nothing fits)
int best_warps_per_block(const MechDev &m, int lu_precision, int driver, int regs);
// Warps (cells) per SM of a persistent batch, of `full` that fit in a block, in
// groups of `couple`.  A batch with fewer cells than that spreads evenly, one block
// of ceil(units / SMs) cells or groups on every SM, since a cell runs the faster the
// fewer share its SM (72/186, first solve of 301 cells: 5.5 ms against 7.3 ms as 26
// full blocks of 12).  A few cells per warp later the batch still lasts about as
// long as its longest cells; up to 24 cells per SM `narrow` batches take two warps
// for each of the SM's four FP64 units, up to 36 ten warps.  ms of a first solve /
// repeated / running, by warps per SM:
//   72/186 (12 fit)   2,048 cells  12: 8.5/9.1/2.0    8: 7.7/7.8/1.8   10: 8.0/8.2/1.8
//                     3,001 cells  12: 9.0/9.3/3.1    8: 8.2/8.1/2.7   10: 8.7/8.8/2.8
//                     5,000 cells  12: 12.3/11.5/2.7  8: 12.5/11.1/2.4 10: 12.3/10.6/2.6
//   50/130 (12 fit)   3,000 cells  12: 7.0/7.4/1.7    8: 7.0/6.4/1.8   10: 7.1/6.8/1.7
// Never below that: with one warp a unit stands idle while it waits (100/260, where 8 fit: 1,700 cells 8: 11.9/9.3/2.4,
// 5: 13.1/8.9/2.5; 2,400 cells 8: 13.2/12.7/2.9, 5: 15.4/13.3/3.0; 128/330, where 4
// fit: 1,000 cells 4: 62.4/55.7/4.3, 2: 66.5/54.0/5.1).
constexpr int NARROW_WARPS = 8, NARROW_WARPS_MORE = 10;      // up to 24, up to 36 cells per SM
inline int shape_warps(int full, int couple, int64_t n_cells, int n_sm, bool narrow) {
  const int64_t units = (n_cells + couple - 1) / couple;
  const int64_t per_sm = (units + n_sm - 1) / n_sm * couple;
  if (per_sm < full) return (int)per_sm;
  if (narrow && per_sm <= 24) return full < NARROW_WARPS ? full : NARROW_WARPS;
  if (narrow && per_sm <= 36) return full < NARROW_WARPS_MORE ? full : NARROW_WARPS_MORE;
  return full;
}
// launch shape of a batch of n_cells in groups of `couple` whose caller gave
// neither cells per block nor blocks per SM (0: nothing fits)
void auto_shape(const MechDev &m, int lu_precision, int driver, int regs, int couple, bool record, int64_t n_cells,
                int *warps_per_block, int *blocks_per_sm);
// diagnostic: mode 0 out = f(y); mode 1 out = (I - c J(y))^{-1} b   (all [S][C] device arrays)
cudaError_t launch_probe(const MechDev &M, const CellsDev &C, int lu_precision, int mode, double c, const double *y,
                         const double *b, double *out, cudaStream_t stream);

// discrete adjoint: replay (exact steps, y rows), backward sweep, theta reduction
cudaError_t launch_adjoint(const MechDev &m, const CellsDev &c, const AdjDev &a, cudaStream_t stream);
cudaError_t launch_tangent(const MechDev &m, const CellsDev &c, const TanDev &t, cudaStream_t stream);
// diagnostic: out[i] = the solve kernels' FP64 reciprocal of x[i] (device arrays)
cudaError_t launch_recip_probe(const double *x, double *out, int64_t n, cudaStream_t stream);
// diagnostic: out[g] = the solve kernels' warp sum of x[32 g .. 32 g + 31] (device arrays)
cudaError_t launch_wsum_probe(const double *x, double *out, int64_t n_groups, cudaStream_t stream);
// *acc += the number of nonzero flags among flag[0..n)
cudaError_t launch_count_flags(const int *flag, int64_t n, unsigned long long *acc, cudaStream_t stream);
// deriv.cu: derivative-only kernels for comparing designs.  kt[R][C] rate
// constants of the batch (launch_rates fills it); y, f [S][C] on the device.
cudaError_t launch_rates(const MechDev &m, const CellsDev &c, double *kt, cudaStream_t stream);
cudaError_t launch_deriv_design(const MechDev &m, const CellsDev &c, int design, const double *kt, const double *y,
                                double *f, cudaStream_t stream);
// kernels.cu: this library's design, without atomics (tiles of 32 cells, one lane per
// cell; the compiled f program, one warp per cell, for the rest)
cudaError_t launch_deriv_gather(const MechDev &m, const CellsDev &c, const double *kt, const double *y, double *f,
                                cudaStream_t stream);

// sets the thread-local message returned by chem_last_error()
void set_last_error(const std::string &msg);

// noalloc.cu: the staging counters of chem_solve_step_noalloc's last call on
// the current device (read on stream, which is then synchronised); a CHEM_*
// return code
int noalloc_stage_counts(int64_t *fallbacks, int64_t *unfinished, cudaStream_t stream);

}  // namespace chemgpu

// opaque handle of include/chemgpu.h
struct chem_mech {
  chemgpu::Mechanism m;
};
