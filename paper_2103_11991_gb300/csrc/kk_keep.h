// Sizes of what a symbolic call keeps of its wide rows, within a budget of bytes.
// Plain arithmetic, so that it is tested on the host over all sizes.
#pragma once

#include <algorithm>
#include <cstdint>

namespace kk {

struct KeepSizes {
  long long rows;       // rows of A
  long long b_rows;     // rows of B
  long long wide_rows;  // rows that may be kept
  long long slot_bytes;     // bits and chunk table of a kept row
  long long slot_tasks;     // chunk tasks that a kept row needs whatever its columns (0: no tasks)
  long long column_tasks;   // further tasks of all rows together, by their columns
  long long long_rows;      // rows of B worth an index, at most
  long long index_bytes;    // an indexed row's positions
};
struct KeepPlan {
  long long slots, tasks, index_rows;
};
constexpr long long kTaskBytes = 8, kMapBytes = 4;  // per task; per row of A, row of B and indexed row

inline long long keep_bytes(const KeepSizes& s, const KeepPlan& p) {
  return p.slots * s.slot_bytes + p.tasks * kTaskBytes + s.rows * kMapBytes +
         (s.slot_tasks > 0 ? s.b_rows * kMapBytes + p.index_rows * (s.index_bytes + kMapBytes) : 0);
}

// No more than wide_rows slots, their tasks and an index of B's long rows; where the
// budget is short, the index and the tasks by columns get a quarter each at most
// (rows without an index are searched, rows whose tasks do not fit are not kept), and
// the slots what is left.  No slots: nothing is kept.
inline KeepPlan keep_plan(long long budget, const KeepSizes& s) {
  KeepPlan p{0, 0, 0};
  const bool chunks = s.slot_tasks > 0;
  long long left = budget - s.rows * kMapBytes - (chunks ? s.b_rows * kMapBytes : 0);
  if (left <= 0) return p;
  if (chunks) {
    p.index_rows = std::min(std::min(s.long_rows, s.b_rows), left / 4 / (s.index_bytes + kMapBytes));
    p.tasks = std::min(s.column_tasks, left / 4 / kTaskBytes);
    left -= p.index_rows * (s.index_bytes + kMapBytes) + p.tasks * kTaskBytes;
  }
  p.slots = std::min(s.wide_rows, left / (s.slot_bytes + s.slot_tasks * kTaskBytes));
  p.slots = std::min(p.slots, 0x7fffffffll);
  p.tasks = std::min(p.tasks + p.slots * s.slot_tasks, 1ll << 28);
  return p;
}

}  // namespace kk
