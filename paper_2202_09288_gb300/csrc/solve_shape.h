// solve_shape.h -- how a level of the solves is launched (host only, no CUDA).
#pragma once

#include <algorithm>
#include <cstdint>

namespace chol {

// Form of a level of a factor that keeps Y (ntasks tasks of nsup supernodes), and right-hand
// sides per CTA.  kNarrow while the tasks fit in one wave at one CTA per SM (its footprint is
// ~115 KB at width 64) and, with several right-hand sides, do not fill every SM with FP64 work
// (then the split form shares the product with Y); kSplit from two tasks per supernode on.
// NR: the fewest per CTA with which the tasks times the groups still fit (an idle SM costs
// nothing, the panel's further reads come from L2) -- for kNarrow, as far as there are
// arrival counters; otherwise the fewest groups of at most 16, evenly filled.
enum SolveMode { kLeaf, kNarrow, kSplit };
constexpr int kWave = 152;
constexpr int kNrList[] = {1, 2, 4, 8, 12, 16};
struct SolveShape {
  int mode, nr, groups;
  int bwd_groups;  // groups per backward launch (a divisor of groups: all of them or one)
};
inline int even_nr(int nrhs) {
  const int groups = (nrhs + 15) / 16, per = (nrhs + groups - 1) / groups;
  for (int nr : kNrList)
    if (nr >= per) return nr;
  return 16;
}
inline int fill_nr(int nrhs, int units, int64_t limit) {
  for (int nr : kNrList)
    if (nr >= nrhs || (int64_t)units * ((nrhs + nr - 1) / nr) <= limit) return nr;
  return even_nr(nrhs);
}
// counters: ints of the backward's arrival array, at least one per supernode of the factor.  A
// backward launch of one group counts on its supernodes' own counters; one of several groups on
// ntasks per group, which only fits where the array is that long (a flat tree of ~100 supernodes
// and 17 or more right-hand sides, two groups whatever NR, is longer: a launch per group).
// kSplit counts nothing.
inline SolveShape solve_shape(int nrhs, int ntasks, int nsup, int64_t counters) {
  const bool split = ntasks >= 2 * nsup && (ntasks > kWave || (int64_t)ntasks * nrhs > 4 * kWave);
  const int mode = split ? kSplit : ntasks <= kWave ? kNarrow : kLeaf;
  const int nr = mode == kSplit    ? fill_nr(nrhs, ntasks, 2 * kWave)
                 : mode == kNarrow ? fill_nr(nrhs, ntasks, std::min<int64_t>(kWave, counters))
                                   : even_nr(nrhs);
  const int groups = (nrhs + nr - 1) / nr;
  const bool together =
      mode == kSplit || (mode == kNarrow && (int64_t)ntasks * groups <= counters);
  return {mode, nr, groups, together ? groups : 1};
}

}  // namespace chol
