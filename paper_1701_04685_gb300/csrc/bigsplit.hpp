// Axis lengths of the cluster kernel's single-warp line transforms (bigfft.cuh).
#pragma once

#include "gensplit.hpp"

namespace fh {

// the split of an axis for warp_two_step: R1 = 0 none, R1 = 1 a line per lane
struct LineSplit {
  int R1, R2;
  unsigned m1, m2;   // lane / R = umulhi(lane, m)
};
inline LineSplit line_split(int N) {
  LineSplit s{};
  if (N >= 2 && N <= 16) {
    s.R1 = 1;
    s.R2 = N;
  } else if (!gen_split(N, false, &s.R1, &s.R2)) {   // radices to 16: 16 warps' registers hold them
    s.R1 = s.R2 = 0;
    return s;
  }
  s.m1 = s.R1 > 1 ? (unsigned)((0x100000000ull + s.R1 - 1) / s.R1) : 0u;
  s.m2 = (unsigned)((0x100000000ull + s.R2 - 1) / s.R2);
  return s;
}

}  // namespace fh
