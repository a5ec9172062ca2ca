// Option defaults and the mapping from spchol_options to plan parameters,
// shared by the GPU library and the host-only library.
#pragma once
#include <algorithm>
#include <cstring>

#include "../../include/spchol.h"
#include "plan.hpp"

namespace spchol {

constexpr int kSolveTileRows = 64;  // rows per solve tile below the near-root band (staged in 32-row chunks)
constexpr int kTrsmTileRows = 64;
constexpr int kFp64TcMinWidth = 16;
// W panels (PlanParams::w_depth) of a single matrix, by default.  Factorization
// + solve, ms, by depth 32 / 64 / 96 / 128: 64^3 with 8 right-hand sides 383.0 +
// 14.5 / 383.2 + 13.8 / 384.2 + 13.1 / 385.6 + 12.6, 27-point 48^3 with FP32
// panels 12.48 + 7.55 / 12.53 + 6.88 / 13.00 + 6.59 / 13.06 + 6.55, 33 x 41 x
// 37 with 16 17.8 + 4.49 / 18.0 + 3.95 / 18.2 + 3.83 / 18.1 + 3.83, 40^3 28.4 +
// 3.94 / 28.6 + 3.51 / 29.0 + 3.29 / 28.9 + 3.27: 64 is the best of one
// factorization and one solve.
constexpr int kWDepth = 64;
// Where the device memory does not hold that many levels' W (by 64^3 66 MB
// beside a factor of 1.3 GB, but by 40^3 83 beside 171 and by 31^3 51 beside 58;
// 32 levels take 17 MB of all three): the next depth an analysis takes.
constexpr int kWDepthLow = 32;

inline void default_options(spchol_options* o) {
  std::memset(o, 0, sizeof(*o));
  o->precision = SPCHOL_FP64;
  o->max_width = 64;
  o->relax_zeros = 4;
  o->tile_rows = 0;
  o->ctas_per_sm = 0;
  o->deterministic = 0;
  o->wait_budget_ns = 2000000000LL;
  o->ir_max_iter = 10;
  o->ir_tol = 1e-12;
  o->fault_inject = 0;
  o->profile = 0;
  o->solve_tile_rows = 0;
  o->sched = 0;
  o->dev_alloc = nullptr;
  o->dev_free = nullptr;
  o->alloc_ctx = nullptr;
  o->solve_w_depth = 0;
}

inline bool options_valid(const spchol_options& o) {
  const bool tc = o.precision == SPCHOL_TF32 || o.precision == SPCHOL_TF32X3 || o.precision == SPCHOL_FP64_TC;
  return o.precision >= SPCHOL_FP64 && o.precision <= SPCHOL_FP64_TC && o.max_width >= 1 &&
         o.max_width <= (tc ? 64 : 128) &&
         o.relax_zeros >= 0 && o.wait_budget_ns > 0 && o.ir_max_iter >= 0 && o.tile_rows >= 0 && o.tile_rows <= 64 &&
         o.ctas_per_sm >= 0 && o.fault_inject >= 0 && o.fault_inject <= 1 && o.deterministic >= 0 &&
         o.deterministic <= 2 &&
         o.profile >= 0 && o.profile <= 2 && o.sched >= 0 && o.sched <= 1 &&
         (o.solve_tile_rows == 0 || (o.solve_tile_rows >= 8 && o.solve_tile_rows <= 256)) &&
         (o.dev_alloc == nullptr) == (o.dev_free == nullptr) && o.solve_w_depth >= -1;
}

inline PlanParams params_from(const spchol_options& o) {
  PlanParams p;
  p.max_width = std::min(std::max(o.max_width, 1), 128);
  p.relax_zeros = std::max(o.relax_zeros, 0);
  p.tile_rows = o.tile_rows > 0 ? o.tile_rows : 64;
  if (o.precision == SPCHOL_TF32 || o.precision == SPCHOL_TF32X3) p.tc_min_width = 1;  // every tile on TF32
  if (o.precision == SPCHOL_FP64_TC) {
    // panels of at least 16 columns carry almost all update work and go to the
    // tensor cores (measured on the 64^3 Laplacian: 201 ms against 210 ms with
    // 32); narrower ones keep DFMA tiles, whose cost scales with size
    p.tc_min_width = kFp64TcMinWidth;
    p.tc_tile_rows = 64;  // the BF16-split tile keeps 64 rows of digits in shared memory
    p.slice_fp64 = true;
  }
  p.trsm_rows = kTrsmTileRows;
  if (o.precision != SPCHOL_FP64) p.level_trsm = 0.3;
  if (o.precision == SPCHOL_FP32) p.level_tiles = 1.0;
  p.fifo = o.sched == 1;
  p.solve_rows = o.solve_tile_rows > 0 ? o.solve_tile_rows : kSolveTileRows;
  p.w_depth = o.solve_w_depth > 0 ? o.solve_w_depth : o.solve_w_depth == 0 ? kWDepth : 0;
  if (o.deterministic) {
    p.deterministic = true;
    p.fanin = o.deterministic == 2;
    p.subtree_flops = 0.0;
    p.w_depth = 0;  // the solves keep the chains of diagonal tasks and tiles
  }
  return p;
}

}  // namespace spchol
