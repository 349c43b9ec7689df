// Axis lengths of the two-step passes of general lengths (genpass.cuh).
#pragma once

namespace fh {

// the split N = R1 R2 with 4 <= R1 <= R2 <= 16 and the smallest R2 (the work of
// the two steps is most even); false where there is none (primes, N < 16, N > 256)
inline bool gen_split(int N, int* R1, int* R2) {
  for (int r2 = 4; r2 <= 16; ++r2)
    if (N % r2 == 0 && N / r2 >= 4 && N / r2 <= r2) {
      *R1 = N / r2;
      *R2 = r2;
      return true;
    }
  return false;
}

}  // namespace fh
