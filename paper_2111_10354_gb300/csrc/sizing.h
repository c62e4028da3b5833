// Sizes that the host chooses from numbers alone (no CUDA here, so that they are tested without a GPU).
#pragma once
#include <stddef.h>

namespace hisq {

// Iterations per group of the multi-shift CG, `most` or a power of two below it: each needs a residual buffer of
// per_slot bytes. What a solve before this one holds (held bytes) costs nothing more; a longer group replaces it and
// has to leave the verification that follows its room: verify bytes, of which verify_held are allocated already.
// Counting what is held makes solves that follow one another take the same length: the first one's choice s satisfies
// s per_slot + verify <= free, 2 s does not, and neither changes once both buffers are taken out of free.
inline int ms_group_length(int most, size_t per_slot, size_t held, size_t verify, size_t verify_held, size_t free_b) {
  const size_t reserve = verify > verify_held ? verify - verify_held : 0;
  int s = most;
  while (s > 1 && s * per_slot > held && s * per_slot + reserve > free_b + held) s /= 2;
  return s;
}

}  // namespace hisq
