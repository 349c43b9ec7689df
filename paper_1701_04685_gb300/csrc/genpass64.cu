// The two-step passes of general lengths (genpass.cuh) in FP64.
#include <algorithm>

#include "genpass.cuh"

namespace fh {

int gen_rows_per_block(double, int nv, int L, long long rows) {
  return nv == 3 ? gen_rb<double, 3>(L, rows) : gen_rb<double, 6>(L, rows);
}

cudaError_t gen_col_prepare(double, int nv, int N) {
  return nv == 3 ? gen_col_prepare_t<double, 3>(N) : gen_col_prepare_t<double, 6>(N);
}
cudaError_t gen_row_prepare(double, const GridInfo& g, int rb) {
  return g.nv == 3 ? gen_row_prepare_t<double, 3>(g, rb) : gen_row_prepare_t<double, 6>(g, rb);
}

cudaError_t gen_col(int mode, const GridInfo& g, int N, const double2* tw, double2* S, const double* G, const LoadState* st,
                    long long stride, int nload, cudaStream_t stream) {
  return g.nv == 3 ? gen_col_t<double, 3>(mode, g, N, tw, S, G, st, stride, nload, stream)
                   : gen_col_t<double, 6>(mode, g, N, tw, S, G, st, stride, nload, stream);
}

cudaError_t gen_row(bool first, bool kinv, const GridInfo& g, const double2* tw, double* E, double2* S, const uint8_t* phase,
                    const double* dC, Control* ctl, LoadState* st, double* partials, double* hist, int nload, int rb, double* Wout,
                    const double* Yaux, const double* Cfld, cudaStream_t stream) {
  return g.nv == 3 ? gen_row_t<double, 3>(first, kinv, g, tw, E, S, phase, dC, ctl, st, partials, hist, nload, rb, Wout, Yaux,
                                       Cfld, stream)
                   : gen_row_t<double, 6>(first, kinv, g, tw, E, S, phase, dC, ctl, st, partials, hist, nload, rb, Wout, Yaux,
                                       Cfld, stream);
}

CheckUnit check_unit_gen64() { return {check_take, check_selftest}; }

}  // namespace fh
