// Launch sizes that have to hold on any device, for host code and its tests.
#pragma once

#include <algorithm>

namespace relres {

// Blocks of a cooperative launch over `work` items on a device with `sms`
// multiprocessors that each hold `per_sm` of its blocks: all of them have to be
// resident at once, and none of them needs more than one item.
inline int cooperative_blocks(int work, int sms, int per_sm) {
  return std::max(1, std::min(work, sms * per_sm));
}

}  // namespace relres
