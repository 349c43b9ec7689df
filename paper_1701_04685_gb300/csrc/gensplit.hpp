// Axis lengths of the two-step passes of general lengths (genpass.cuh).
#pragma once

#include <cstddef>

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

// A line of R1 R2 points in shared memory: row k1 at offset (R2 | 1) k1, so that its
// stride is odd; the line stride is the next one that leaves `rest` mod 16.
inline int gen_row_stride(int R2) { return R2 | 1; }
inline int gen_line_stride(int R1, int R2, int rest) {
  const int need = R1 * gen_row_stride(R2);
  return need + ((rest - need) % 16 + 16) % 16;
}
// a column tile: line stride 16 / ct mod 16 (FP64: 2), so that the lanes of an access
// phase fall on distinct banks
inline int gen_col_stride(int R1, int R2, bool fp32, int ct) { return gen_line_stride(R1, R2, fp32 ? 16 / ct : 2); }

// Columns per block of the column pass along an axis of N points, 0 where the pass does
// not apply (no split, or a tile of its twiddles and n_v ct lines that no block can
// hold).  Eight in FP32 3-D, four where eight do not fit (N > 512: 576, 640, 768, 1024),
// in FP64 and in 2-D.
constexpr size_t kGenColSmem = 226 * 1024;   // of the 227 KB a block may ask for; the rest is the kernel's own
inline size_t gen_col_bytes(int N, bool fp32, int nv, int ct) {
  int R1 = 0, R2 = 0;
  if (!gen_split(N, fp32, &R1, &R2)) return 0;
  return (size_t)(N + nv * ct * gen_col_stride(R1, R2, fp32, ct)) * (fp32 ? 8 : 16);
}
inline int gen_columns(int N, bool fp32, int nv) {
  int R1 = 0, R2 = 0;
  if (!gen_split(N, fp32, &R1, &R2)) return 0;
  for (int ct = fp32 && nv == 6 ? 8 : 4; ct >= 4; ct /= 2)
    if (gen_col_bytes(N, fp32, nv, ct) <= kGenColSmem) return ct;
  return 0;
}

}  // namespace fh
