// The two-step passes of general lengths (genpass.cuh) in FP64.
#include <algorithm>

#include "genpass.cuh"

namespace fh {

int gen_rows_per_block(double, int L) { return gen_rb<double>(L); }

cudaError_t gen_col(int mode, const GridInfo& g, int N, const double2* tw, double2* S, const double* G, const LoadState* st,
                    long long stride, int nload, cudaStream_t stream) {
  return gen_col_t<double>(mode, g, N, tw, S, G, st, stride, nload, stream);
}

cudaError_t gen_row(bool first, bool kinv, const GridInfo& g, const double2* tw, double* E, double2* S, const uint8_t* phase,
                    const double* dC, Control* ctl, LoadState* st, double* partials, double* hist, int nload, double* Wout,
                    const double* Yaux, cudaStream_t stream) {
  return gen_row_t<double>(first, kinv, g, tw, E, S, phase, dC, ctl, st, partials, hist, nload, Wout, Yaux, stream);
}

cudaError_t gen_take_check64(CheckRecord* rec) {
  *rec = CheckRecord{};
#ifdef FH_CHECKED
  cudaError_t e = cudaMemcpyFromSymbol(rec, g_check, sizeof(*rec));
  if (e == cudaSuccess && rec->count != 0ull) {
    const CheckRecord zero{};
    e = cudaMemcpyToSymbol(g_check, &zero, sizeof(zero));
  }
  return e;
#else
  return cudaSuccess;
#endif
}

}  // namespace fh
