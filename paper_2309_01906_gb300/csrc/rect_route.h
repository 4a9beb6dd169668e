// rect_route.h — which kernel takes a rectangular plan's memory-reading rows: the
// launch (rect_launch.cuh) and the plan's description ask the same questions.
#pragma once

#include "hp_internal.h"

namespace hp {

constexpr int64_t kRowsMaxR = int64_t(1) << 22;   // rect_rows_kernel: 32-bit offsets within a warp's rows
constexpr int kThreadRowsMin = 5, kThreadRowsMax = 64;   // rect_thread_rows_kernel: elements per row
constexpr int kFlatThreads = 256;                 // rect_flat_kernel: threads per CTA, at most

inline bool reads_memory(const NestPlan& p) { return p.body == HP_BODY_LOAD || p.body == HP_BODY_DOT_BCAST; }

// Which kernel folds whole rows (rect_rows_kernel, rect_thread_rows_kernel)?
// aligned: does the input start on 16 bytes?
enum RowsKind { ROWS_NONE = 0, ROWS_TEAM = 1, ROWS_THREAD = 2 };
inline RowsKind rows_kind(const NestPlan& p, bool aligned) {
  const RectPlan& rp = p.rp;
  if (!reads_memory(p) || rp.team != TEAM_LANES || rp.nv != 1 || rp.vstride[0] != 1 || rp.G != 1 || rp.split || rp.R < 1 ||
      rp.R > kRowsMaxR)
    return ROWS_NONE;
  const bool dot = p.body == HP_BODY_DOT_BCAST, comp = p.prec == HP_F32_COMP && p.op == HP_RED_SUM;
  const bool wide = comp || p.prec == HP_I64;   // 8-byte accumulators
  // vectors of plain rows from 16 elements on load whole sectors anyway (2^25
  // elements in rows of 16, int64: 27 us in rect_lanes_kernel, 28 through shared memory)
  const bool sectors = rp.V == 4 && rp.R >= 16 && !dot && !comp;
  // one or two lanes a row: blocks of 32 rows are copied 16 bytes at a time
  if (rp.R >= (wide && dot && rp.V == 4 ? 4 : kThreadRowsMin) && aligned && !sectors &&
      (rp.L == 1 ? rp.R <= 32   // one lane: every slot coefficient is 0
                 : rp.L == 2 && rp.V == 1 && rp.cl[0] == 1 && rp.grp_lanes >= 2 && rp.R <= kThreadRowsMax))
    return ROWS_THREAD;
  return rp.L > 1 || rp.R < 5 ? ROWS_TEAM : ROWS_NONE;
}

// Does an item of this block-team plan lie in consecutive elements that
// rect_flat_kernel can fold?  It also takes plain reductions of long rows from the
// cp.async pipeline (2^26 elements, f32 / compensated / int64: rows of 4096 44, 54 and
// 47 us there and 38, 44 and 39 here, 6400 51, 62, 59 and 39, 44, 39, 8192 43, 45, 44
// and 40, 38, 37); the pipeline stays for dot products (compensated, 7168: 47 there,
// 53 here) and 64-bit comparisons (5344: 50 and 52), for rows that a round of it
// holds several of, and for other levels.
inline bool flat_plan(const NestPlan& p) {
  const RectPlan& rp = p.rp;
  const bool leave = p.body == HP_BODY_LOAD && !(p.prec == HP_I64 && p.op != HP_RED_SUM);
  return reads_memory(p) && rp.team == TEAM_BLOCK && rp.C == 1 && rp.W <= kFlatThreads / 32 && rp.nv == 1 && rp.vstride[0] == 1 &&
         (!rp.pipe || (leave && rp.R >= 4096)) && rp.R >= 1 &&
         (rp.G > 1 ? rp.split && rp.tile < (int64_t(1) << 30) : rp.R < (int64_t(1) << 30));
}

}  // namespace hp
