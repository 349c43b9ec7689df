// The two-step passes of general lengths (genpass.cuh) in FP32.
#include <algorithm>

#include "genpass.cuh"

namespace fh {

int gen_rows_per_block(float, int nv, int L, long long rows) {
  return nv == 3 ? gen_rb<float, 3>(L, rows) : gen_rb<float, 6>(L, rows);
}

cudaError_t gen_col_prepare(float, int nv, int N) {
  return nv == 3 ? gen_col_prepare_t<float, 3>(N) : gen_col_prepare_t<float, 6>(N);
}
cudaError_t gen_row_prepare(float, const GridInfo& g, int rb) {
  return g.nv == 3 ? gen_row_prepare_t<float, 3>(g, rb) : gen_row_prepare_t<float, 6>(g, rb);
}

cudaError_t gen_col(int mode, const GridInfo& g, int N, const float2* tw, float2* S, const float* G, const LoadState* st,
                    long long stride, int nload, cudaStream_t stream) {
  return g.nv == 3 ? gen_col_t<float, 3>(mode, g, N, tw, S, G, st, stride, nload, stream)
                   : gen_col_t<float, 6>(mode, g, N, tw, S, G, st, stride, nload, stream);
}

cudaError_t gen_row(bool first, bool kinv, const GridInfo& g, const float2* tw, float* E, float2* S, const uint8_t* phase,
                    const float* dC, Control* ctl, LoadState* st, double* partials, double* hist, int nload, int rb, float* Wout,
                    const float* Yaux, const float* Cfld, cudaStream_t stream) {
  return g.nv == 3 ? gen_row_t<float, 3>(first, kinv, g, tw, E, S, phase, dC, ctl, st, partials, hist, nload, rb, Wout, Yaux,
                                       Cfld, stream)
                   : gen_row_t<float, 6>(first, kinv, g, tw, E, S, phase, dC, ctl, st, partials, hist, nload, rb, Wout, Yaux,
                                       Cfld, stream);
}

CheckUnit check_unit_gen32() { return {check_take, check_selftest}; }

}  // namespace fh
