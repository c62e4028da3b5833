// Sizes that the host chooses from numbers alone (no CUDA here, so that they are tested without a GPU).
#pragma once
#include <stddef.h>

#include <algorithm>

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

// Ways to cut the vectors of a Dslash into launches of at most gmax vectors.
enum LaunchCut {
  CUT_FULL = 0,  // groups of gmax, and what is left in one launch
  CUT_EVEN = 1,  // groups of nearly equal size
  CUT_POW2 = 2,  // groups of gmax, and what is left in powers of two
};

// Vectors of the next launch when `left` are left.
inline int next_group(int cut, int left, int gmax) {
  if (cut == CUT_EVEN) {
    const int groups = (left + gmax - 1) / gmax;
    return (left + groups - 1) / groups;
  }
  if (left >= gmax || cut == CUT_FULL) return std::min(left, gmax);
  int p = 1;
  while (2 * p <= left) p *= 2;
  return p;
}

// The ways that differ for nrhs vectors, CUT_FULL first; CUT_POW2 only where asked for. Returns how many.
inline int launch_cuts(int nrhs, int gmax, bool pow2, int (&cuts)[3]) {
  int n = 0;
  for (int c : {CUT_FULL, CUT_EVEN, CUT_POW2}) {
    if (c == CUT_POW2 && !pow2) continue;
    bool fresh = true;
    for (int k = 0; k < n && fresh; ++k) {
      int a = nrhs, b = nrhs;
      while (a > 0 && a == b) {
        a -= next_group(cuts[k], a, gmax);
        b -= next_group(c, b, gmax);
      }
      fresh = a != b;
    }
    if (fresh) cuts[n++] = c;
  }
  return n;
}

}  // namespace hisq
