// schedule_view.cpp -- reads a handle's host-side schedule for the tests that
// check it without a GPU (tests/test_schedule.py).
#include "internal.h"

// TRSM tasks of the blocked path as (supernode, first column of the step, first
// row, supernode's columns, supernode's rows). Returns their number; out may be null.
extern "C" int64_t view_trsm(const chol_handle* h, int32_t* out) {
  int64_t k = 0;
  for (const LevelPlan& P : h->levels)
    for (const StepRange& s : P.steps)
      for (int32_t i = s.trsm_b; i < s.trsm_b + s.trsm_n; ++i, ++k)
        if (out) {
          const TileTask& t = h->trsm_tasks[i];
          const SnodeDev& d = h->snodes[t.J];
          const int32_t v[5] = {t.J, t.k0, t.r0, d.s, d.len};
          for (int c = 0; c < 5; ++c) out[5 * k + c] = v[c];
        }
  return k;
}

// Rows of one binary64 TRSM task.
extern "C" int32_t view_trsm_rows() { return kTrsmRowsHost / 2; }
