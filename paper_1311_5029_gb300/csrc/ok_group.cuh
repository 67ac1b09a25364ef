// How many pairs of a training batch go through the kernels together when memory is short.
#pragma once

namespace okgb {

// The group's new size: at most `want` pairs, at least the `have` whose buffers there are already.  alloc(q) gets buffers
// for q pairs beside those and says whether it could.  A group that does not fit is halved; `most` remembers
// what did (0: nothing has been refused), so that later steps neither ask again nor give up what they have.
template <typename Alloc>
int grow_group(int want, int have, int& most, Alloc&& alloc) {
  if (most > 0 && want > most) want = most;
  for (int q = want; q > have; q /= 2) {
    if (alloc(q)) return q;
    most = q / 2 > have ? q / 2 : have;
  }
  return have;
}

}  // namespace okgb
