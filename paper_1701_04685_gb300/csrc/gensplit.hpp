// Axis lengths of the two-step passes of general lengths (genpass.cuh).
#pragma once

namespace fh {

// radices with a register DFT (gendft.cuh); those above 16 in FP32 only, whose
// registers hold them
inline bool gen_radix(int r, bool fp32) {
  return (r >= 4 && r <= 16) || (fp32 && (r == 18 || r == 20 || r == 24 || r == 32));
}

// the split N = R1 R2 with R1 <= R2 and the smallest R2 (the work of the two steps
// is most even); false where there is none (primes, N < 16, N > 256 in FP64 or 1024
// in FP32)
inline bool gen_split(int N, bool fp32, int* R1, int* R2) {
  for (int r2 = 4; r2 <= 32; ++r2)
    if (gen_radix(r2, fp32) && N % r2 == 0 && N / r2 <= r2 && gen_radix(N / r2, fp32)) {
      *R1 = N / r2;
      *R2 = r2;
      return true;
    }
  return false;
}

}  // namespace fh
