// The two-step passes of general lengths (genpass.cuh) in FP32.
#include <algorithm>

#include "genpass.cuh"

namespace fh {

int gen_rows_per_block(float, int L) { return gen_rb<float>(L); }

cudaError_t gen_col(int mode, const GridInfo& g, int N, const float2* tw, float2* S, const float* G, const LoadState* st,
                    long long stride, int nload, cudaStream_t stream) {
  return gen_col_t<float>(mode, g, N, tw, S, G, st, stride, nload, stream);
}

cudaError_t gen_row(bool first, bool kinv, const GridInfo& g, const float2* tw, float* E, float2* S, const uint8_t* phase,
                    const float* dC, Control* ctl, LoadState* st, double* partials, double* hist, int nload, float* Wout,
                    const float* Yaux, cudaStream_t stream) {
  return gen_row_t<float>(first, kinv, g, tw, E, S, phase, dC, ctl, st, partials, hist, nload, Wout, Yaux, stream);
}

cudaError_t gen_take_check32(CheckRecord* rec) {
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
