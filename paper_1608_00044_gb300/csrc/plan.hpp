// Host-side analysis result: supernode partition, row structures, storage
// layout and the task graph of the factorization and the solves.
#pragma once
#include <cstdint>
#include <string>
#include <vector>

namespace spchol {

// FP64 tensor-core mode: every FP64 value of L below a diagonal block is split
// into this many 8-bit slices relative to its row's largest magnitude.
constexpr int kSlices = 7;
constexpr int kSliceBits = 8;

// One update tile U(s, t): rows [row0, row0 + rowlen) of source panel s (indices
// into s's row list) times the rows [seg0, seg0 + seglen) of s that fall inside
// target panel t's columns (Section III-A, task U; Section IV, task T_{s,t}).
struct UTask {
  int32_t s, t, seg0, seglen, row0, rowlen;
  int64_t rel;  // offset of the tile's relative row indices (rowlen of them) in the relative-index array
};

struct PlanParams {
  int max_width = 64;    // W (Section III-B caps supernodes at 150 columns)
  int relax_zeros = 4;   // amalgamation budget per column
  int tile_rows = 64;    // rows per update tile
  int trsm_rows = 128;   // rows per panel-solve tile
  int solve_rows = 128;  // rows per triangular-solve tile
  // Panels within top_depth of the root of the panel etree (the chains of the
  // top separators: the critical path): their update tiles into the etree
  // parent go ahead of the others, and their solve tiles are shorter.
  int top_depth = 128;
  // Rows per update tile: the panels of one level (distance to the root) take
  // the largest of tile_rows, 32 and 16 that still gives the level level_tiles
  // tiles per CTA (kPlanCtas); rows per panel-solve tile:
  // of trsm_rows, 32 and 16, level_trsm tiles.  A level with fewer is on the
  // critical path and its tiles have to spread; one with more only pays each
  // tile's claim, staging and publishing.  level_tiles 0: by the size of the
  // problem (FP64 tiles), 8 (flops / 2.4e10)^0.4 within 4 .. 32.  Measured, ms
  // of the FP64 factorization by level_tiles (with 16 rows within 128 levels of
  // the root and tile_rows below, the rule before: 10.6, 20.5, 33.2, 76.4,
  // 102.7 and 387.2):
  //                 4      6      8      12     16     24
  //   31 x 34 x 29  9.81   9.54   9.91  10.49  10.71
  //   33 x 41 x 37 19.03  18.25  18.32  18.98  19.92
  //   40^3         30.4   29.3   28.8   29.7   30.7
  //   27-pt 48^3   78.1   77.0   76.3   75.0   74.6
  //   50^3         98.0   97.8   96.8   94.9   95.8
  //   64^3        390.6  390.6  390.0  388.3  386.9
  // FP32 tiles are 5 us of arithmetic to 5 us of the rest and want fewer (27-pt
  // 48^3 by 0.5 / 1 / 2 / 4 / 8: 12.58 / 12.48 / 12.50 / 12.60 / 13.03 ms,
  // 17.9 before; 40^3 9.7 up to 4, 15.7 before), as do the panel-solve tiles
  // beside tensor-core updates (64^3 FP64_TC by 0.3 / 1 / 3: 152.3 / 155.1 /
  // 159.0 ms).
  double level_tiles = 0.0;
  double level_trsm = 1.0;
  int top_solve_rows = 32;  // rows per triangular-solve tile of those panels
  // Tensor-core update tiles: source panels at least tc_min_width wide (0 =
  // none) use tc_tile_rows-row tiles (one MMA M-tile) on the tensor cores.
  int tc_min_width = 0;
  int tc_tile_rows = 128;
  bool slice_fp64 = false;  // FP64 tensor-core mode: split those panels into BF16 digits
  // Subtree tasks: a maximal subtree of the panel etree whose factorization
  // costs at most min(subtree_flops, total flops / 4096) runs as one task
  // (0: none).
  double subtree_flops = 1e6;
  // Deterministic order (the static (target, source) order of Section IV-B):
  // see Plan::u_next.  Subtree tasks are off in this mode.
  bool deterministic = false;
  // Deterministic by fan-in aggregation (the fan-in family of Section II-C, restated
  // for one GPU) instead of the chains: see Plan::fan_ptr.  Implies
  // deterministic (the solves keep their chains).
  bool fanin = false;
  // One FIFO ready ring instead of the two priority rings (spchol_options.sched
  // = 1): the launch gives the high-priority ring no slots, and every push goes
  // to the other ring.  The plan itself is the same.
  bool fifo = false;
  // Panels within w_depth of the root of the panel etree (0: none), outside
  // subtree tasks, at most kWMaxWidth wide and with rows below their diagonal
  // block, also keep W = L21 L11^{-1} (Plan::woff), so that their solve steps
  // need no diagonal task on the chain: see Plan::woff.
  int w_depth = 0;
};

// The CTAs that tile rows and the subtree cut are laid out for, a nominal unit:
// 152 SMs x 5, the resident CTAs of the plain FP64 kernel.  FP32 panels run 6
// per SM, the fan-in kernels 4, FP64_TC 3, TF32 2, and ctas_per_sm can lower
// them; the limits below were measured against this unit in each mode, and with
// ctas_per_sm 1 and 2 (31^3 FP64: factorization 24.2 -> 17.4 and 18.6 -> 11.1
// ms, the rules before -> these).
constexpr int kPlanCtas = 152 * 5;

// In a small problem (at most kFuseFlops), a panel of at most kFuseWidth columns
// with few rows below them (w^2 rows <= kFuseWork, at most kFuseRows) has a
// single panel-solve tile, and its diagonal task solves those rows itself,
// from the L11 it holds in shared memory: on the lower levels a task is mostly
// its fixed costs (a claim, the panel's sizes, staging, publishing: 8 us of
// the 8-column panel's 9), and the chain of a small problem is made of them.
// Factorization before -> now, ms: 24^2 0.224 -> 0.178, 64^2 0.447 -> 0.415, 12^3
// 0.840 -> 0.813, 27-point 20^3 2.29 -> 2.24, 181 x 203 1.59 -> 1.58, 250 x 256
// 2.55 -> 2.50.  Larger ones are bound by their tiles, and the kernel that can
// do it has more registers to spill (31 x 34 x 29 9.23 -> 9.34, 27-point 48^3
// with FP32 panels 12.6 -> 13.1): they keep the kernel without it.
constexpr int kFuseWidth = 32, kFuseRows = 64, kFuseWork = 32 * 32 * 32;
constexpr double kFuseFlops = 1e9;
inline bool fuse_shape(int w, int nb) { return w <= kFuseWidth && nb > 0 && nb <= kFuseRows && w * w * nb <= kFuseWork; }

// Widest panel of a subtree task that runs on one warp (Plan::wsub).
constexpr int kWarpSubW = 32;

// Widest panel that keeps W = L21 L11^{-1} (its packed inverse is staged in
// shared memory by the panel-solve tiles that form W).
constexpr int kWMaxWidth = 64;

// Rows of a target panel are gathered in pieces of at most this many rows.
constexpr int kFanPieceRows = 32;

// One entry of a fan-in gather list: rows [i0, i1) of update tile u fall in the
// piece that owns the list; its columns [j0, j1) are listed (all of the tile's,
// or those in the window of a split gather).
struct FanEnt {
  int32_t u;
  int16_t i0, i1, j0, j1;
};

// One gather task of the fan-in mode: list entries [e0, e1) (gather_entries),
// which add into columns [c0, c1) of piece pc.
struct GatherTask {
  int64_t e0, e1;
  int32_t pc;
  int16_t c0, c1;
};

struct Plan {
  int64_t n = 0;
  int64_t nnz_a = 0;
  std::vector<int64_t> perm;  // final new -> old (input perm refined by a postorder)
  std::vector<int64_t> pinv;  // old -> new

  // exact structure (before amalgamation)
  int64_t nnz_l = 0;
  double flops = 0.0;  // sum of c_j^2
  std::vector<int64_t> colcount;
  std::vector<int32_t> etree;

  // panels (supernodes after amalgamation and the width cap)
  int32_t ns = 0;
  std::vector<int32_t> fcol;    // ns + 1
  std::vector<int32_t> nrows;   // rows incl. the diagonal block
  std::vector<int32_t> ld;      // leading dimension (nrows rounded up to 4)
  std::vector<int64_t> rowoff;  // ns + 1, into rows
  std::vector<int32_t> rows;    // concatenated sorted row lists
  std::vector<int64_t> valoff;  // ns + 1, into the value pool (elements)
  std::vector<int64_t> invoff;  // ns + 1, into the diagonal-block inverse buffer (w x w per panel)
  std::vector<int64_t> sliceoff;  // ns + 1, into the BF16 slice buffer (FP64 tensor-core mode)
  std::vector<int32_t> parent;  // panel etree, -1 at roots
  std::vector<int32_t> snode_of;  // column -> panel
  std::vector<int64_t> a_dest;  // entry e of A's lower CSC -> pool index
  int64_t nnz_l_stored = 0;
  int32_t max_w = 0, max_r = 0;

  // factorization tasks: [0, ns) diagonal factor, then panel-solve tiles, then updates
  std::vector<int32_t> trsm_first, ntrsm, trsm_sn, trsm_rows;  // trsm_rows: tile rows per panel
  std::vector<int32_t> u_first, nu;
  std::vector<UTask> ut;
  std::vector<int32_t> dep_f;  // update tiles targeting each panel
  int64_t n_rel = 0;           // relative row indices of all update tiles (sum of rowlen)
  // Scheduling priority: diagonal and panel-solve tasks, and the first nu_hi[s]
  // update tiles of panel s (those into its etree parent, for panels within
  // top_depth of the root), go to the high-priority ready ring; n_hi_tasks of
  // them in all.  The remaining update tiles go to the other ring.
  std::vector<int32_t> nu_hi;
  // Subtree tasks: task ns + n_trsm + n_u + k factors panels sub_lo[k] ..
  // sub_hi[k] (a whole subtree: panels are numbered in postorder) in order in
  // one CTA; the panel-level tasks of those panels are never scheduled.
  // in_sub[s]: the subtree task of panel s, or -1.
  std::vector<int32_t> sub_lo, sub_hi, in_sub;
  // The subtree tasks whose panels are all at most kWarpSubW columns wide:
  // the FP64 factorization runs each of them on one warp (see wsub in
  // FactorArgs), several side by side in a CTA.
  std::vector<int32_t> wsub;
  double sub_work_frac = 0.0;  // the subtree tasks' share of the factorization's work
  int32_t n_trsm = 0, n_u = 0, n_sub = 0;
  int32_t n_task_ids = 0;      // size of the task id space: ns + n_trsm + n_u + n_sub
  int32_t n_factor_tasks = 0;  // tasks that are scheduled (pushed to a ring) in one factorization
  int32_t n_hi_tasks = 0;

  // solve tasks
  std::vector<int32_t> st_first, nst, st_sn, st_rows;  // st_rows: solve tile rows per panel
  std::vector<int32_t> kid_ptr, kids;  // panel children, CSR
  // precise solve dependencies: the panels whose columns each solve tile's rows
  // fall in (tile -> targets, CSR), the same relation reversed (panel -> tiles),
  // forward counters (tiles touching each panel) and backward tile counters
  // (targets + 1 for "every forward tile of the tile's own panel is done")
  std::vector<int32_t> st_tptr, st_tgt, rt_ptr, rt_tile, fdep0, bdep0;
  int32_t n_st = 0, n_solve_tasks = 0;
  // W panels (PlanParams::w_depth): woff[s] >= 0 is the offset (elements) of
  // panel s's W = L21 L11^{-1} in the W buffer, stored like the panel itself
  // (column-major, leading dimension ld[s], rows w .. nrows-1 used); -1 for the
  // other panels.  The panel-solve tiles of the factorization write W after
  // their L21 rows.  The solves then take, for a W panel s, b_s = the
  // right-hand side rows of s once every forward tile into s has landed:
  //   forward tile k:  y[rows of k] -= W[k] b_s   (ready with b_s, no diagonal task first)
  //   diagonal task:   y_s <- L11^{-T} L11^{-1} b_s, after every forward tile of s has read b_s
  //   backward tile k: y_s -= W[k]^T x[rows of k], after the diagonal task
  // and x_s = y_s once the backward tiles are done (the last one releases the
  // dependents, the role of the backward diagonal task, which never runs):
  // x_s = L11^{-T} (L11^{-1} b_s - L21^T x_below) = A11^{-1} b_s - W^T x_below.
  std::vector<int64_t> woff;
  int64_t n_w = 0;      // elements of the W buffer
  int32_t n_wpan = 0;   // W panels (backward diagonal tasks that never run)
  int32_t levels = 0;   // of the panel tree

  // Deterministic order (params.deterministic; empty otherwise).  The update
  // tiles into each target panel form a chain in (source panel, row tile)
  // order, and a tile becomes ready only when its source's panel-solve tiles
  // and its predecessor in the chain are done, so the scatter-adds into every
  // entry land in one fixed order: u_next (next tile into the same target, -1
  // at the end) and u_dep0 (1 + 1 with a predecessor).  Likewise the forward
  // solve tiles that subtract from each panel's rows chain in tile order
  // (ft_sptr / ft_succ: each tile's successors, one per target panel chain;
  // ft_dep0: 1 for its panel's diagonal solve + its predecessors), and the
  // backward tiles of a panel, which all subtract from that panel's entries,
  // chain in tile order (bdep0 counts the predecessor).
  std::vector<int32_t> u_next, u_dep0, ft_sptr, ft_succ, ft_dep0;

  // Fan-in aggregation (params.fanin; empty otherwise).  Update tile u stores
  // its product, negated, densely (column-major, rowlen rows, seglen columns,
  // lower entries only) at fan_off[u] of a private buffer instead of adding
  // it into the target.  The rows of each target panel are split into pieces:
  // the diagonal block in steps of kFanPieceRows rows, then each panel-solve
  // tile's rows in such steps.  fan_task[k] (k < ns: the diagonal task of
  // panel k; k >= ns: panel-solve tile k - ns) is the first piece of that
  // task's rows, whose pieces are consecutive; fan_ptr / fan_ent list, for
  // every piece in update-tile order, the tiles with rows in it and which.
  // The task that owns a piece adds those buffers into its rows in list
  // order before it factors or solves them, so every entry of L receives
  // its updates in one fixed order, and the update tiles themselves need no
  // order among them.
  std::vector<int64_t> fan_off;   // n_u + 1
  std::vector<int32_t> fan_task;  // ns + n_trsm
  std::vector<int64_t> fan_ptr;   // pieces + 1
  std::vector<FanEnt> fan_ent;
  std::vector<int64_t> pc_values;  // pieces: the values their lists add
  // The solves of the fan-in mode: forward tile k stores its product (its
  // rows x nrhs, negated) at st_zf[k] * nrhs of one buffer and backward tile k
  // its product (its panel's width x nrhs) at st_zb[k] * nrhs of another,
  // instead of adding them into the right-hand sides.  A panel's forward
  // diagonal task adds the forward buffers of the tiles with rows in its
  // columns first, in tile order (its rt_tile list read from the end; rt_rng:
  // those rows of the tile, i0 | i1 << 16; st_roff: the tile's first row in
  // the row lists), and its backward diagonal task adds its own tiles'
  // backward buffers in tile order: every entry of the solution receives its
  // updates in one fixed order -- the order of the static chains.
  // Gather tasks (fan-in mode): one per row piece that receives updates, task
  // id ns + n_trsm + n_u + n_sub + g for g in [gat_first[t], gat_first[t + 1])
  // of panel t, piece gat[g].pc, all made ready when the panel's last update
  // tile lands.  pc_owner[piece]: the task whose rows it holds (t: the
  // diagonal task, ns + k: panel-solve tile k).  The diagonal task waits for
  // its gathers (gdiag0[t] of them; none: it is ready with the updates), each
  // panel-solve tile for the diagonal task and its own gathers (tdep0[k]).
  std::vector<int32_t> gat_first, pc_owner, gdiag0, tdep0;
  std::vector<GatherTask> gat;
  std::vector<FanEnt> gat_ent;  // the tasks' lists once split_gathers has cut them; before, they are the pieces' own (fan_ent)
  int32_t n_gat = 0;
  std::vector<int64_t> st_zf, st_zb;  // n_st + 1
  // the forward gather's record of each rt_tile entry: the tile's buffer (in
  // rows: st_zf), its first listed row's place in the row lists, the tile's
  // rows, its first listed row and how many are listed
  struct SolveFanRec {
    int64_t z, ro;
    int32_t cnt;
    int16_t i0, ni;
  };
  std::vector<SolveFanRec> rt_rec;
  std::vector<int64_t> st_roff;       // n_st
  std::vector<int32_t> rt_rng;        // like rt_tile

  PlanParams params;
};

// Validation error: argument index (1-based) and message.
struct PlanError {
  int arg = 0;
  std::string msg;
};

// Builds the plan.  Returns 0, or -k with err filled for an invalid argument k
// (1 n, 2 colptr, 3 rowind, 4 perm).
int build_plan(int64_t n, const int64_t* colptr, const int32_t* rowind, const int64_t* perm,
               const PlanParams& params, Plan& plan, PlanError& err);

// Replaces every subtree task of more than max_steps steps (a step: a diagonal
// task, a panel-solve tile or an update tile) by the maximal subtrees inside it
// that stay within max_steps; the panels above those become tasks of their
// own.  Not after the warp-level launches have been laid out (Plan::wsub).
void split_subtrees(Plan& plan, int64_t max_steps);

// The lists that Plan::gat's tasks index.
inline const std::vector<FanEnt>& gather_entries(const Plan& P) { return P.gat_ent.empty() ? P.fan_ent : P.gat_ent; }

// Split the gather tasks that add more than max_values values (fan-in mode)
// into column windows of a multiple of 8 columns, each with a list of its own:
// gathers of one piece add into disjoint columns, so every entry still receives
// its updates in the piece's list order.  Every task's list is written to
// Plan::gat_ent, one after another.  A gather adds its tiles one after another,
// and near the root -- 300 tiles and 100,000 values a piece, one panel after
// another, the chip idle -- those were most of the critical path (300 us each).
// Factorization of a 27^3 Laplacian: no split 11.8 ms, at 16384 values 8.6, 8192
// 8.0, 4096 7.8, 2048 7.8 (and more list entries the finer: 0.50, 0.61, 0.71,
// 0.84 and 1.02 million, which the analysis makes).
constexpr int64_t kGatherValues = 8192;
void split_gathers(Plan& plan, int64_t max_values);

// The GPU launch's max_steps: a CTA's average share of all steps (of kPlanCtas)
// over kSubtreeShare.  A subtree task runs its steps one after
// another, so one that holds more than the average share of the whole
// factorization outlasts everything else: the 1e6-flop budget alone left the
// 31 x 34 x 29 Laplacian with 128 tasks of up to 2633 steps (13 of its 19.6
// ms) against an average share of 645.  Measured factorization times (ms) by
// kSubtreeShare, "none" the flop budget alone:
//                          none     2      3      4      8     16
//   64^2 (FP64)            0.556  0.523  0.527  0.531  0.531  0.526
//   181 x 203              2.08   1.73   1.78   1.81   1.86   1.97
//   31 x 34 x 29          19.5   11.29  10.85  10.93  10.92  10.97
//   40^3                  37.5   33.8   33.4   33.1   33.1   33.2
//   40^3, FP32 panels     19.1   15.8   15.5   15.0   14.9   15.0
//   27-point 48^3, FP32   17.94  17.94  17.99  18.04  18.18  18.30
//   27-point 35x31x38, TF32X3 7.15 6.66  6.68   6.72   7.00   7.10
// (the subtrees of 50^3 and 64^3 are within it from 4 and 6 on).
constexpr int kSubtreeShare = 3;
inline int64_t subtree_step_budget(const Plan& P) {
  int64_t total = 0;
  for (int32_t s = 0; s < P.ns; ++s) total += 1 + P.ntrsm[s] + P.nu[s];
  return total / (kPlanCtas * kSubtreeShare);
}

}  // namespace spchol
