#include "batched_schedule.h"

// The default schedule: the levels' group counts in cnt, how often each matrix
// is placed in placed, estimated times of the default, the tree and the equal
// groups in seconds.  Returns the number of levels.
extern "C" int schedule(int batch, const int64_t* m, const int64_t* n, const int* b, int grid, int* cnt, int* placed,
                        double* seconds) {
  const cqr::BSchedule S = cqr::schedule_default(batch, m, n, b, grid);
  for (int l = 0; l < S.lev.n; ++l) cnt[l] = S.lev.cnt[l];
  for (int i : S.order) ++placed[i];
  seconds[0] = S.seconds;
  seconds[1] = cqr::schedule_tree(batch, m, n, b, grid).seconds;
  seconds[2] = cqr::schedule_uniform(batch, m, n, b, grid, cqr::default_group(grid)).seconds;
  return S.lev.n;
}
