// Host side of the two-step passes of general lengths (genpass.cuh), one
// translation unit per precision so that they compile beside the solver.
#pragma once

#include <cuda_runtime.h>

#include "internal.hpp"
#include "kernels.cuh"

namespace fh {

// rows per block of the row pass for rows of L points (gen_split), n_v components
// and the given number of rows over all loads
int gen_rows_per_block(double, int nv, int L, long long rows);
int gen_rows_per_block(float, int nv, int L, long long rows);

// once per solve, before the launches: the kernels' shared-memory limits (allow_smem)
cudaError_t gen_col_prepare(double, int nv, int N);
cudaError_t gen_col_prepare(float, int nv, int N);
cudaError_t gen_row_prepare(double, const GridInfo& g, int rb);
cudaError_t gen_row_prepare(float, const GridInfo& g, int rb);

// pass along an axis of N points with element stride `stride` (modes as line_pass)
cudaError_t gen_col(int mode, const GridInfo& g, int N, const double2* tw, double2* S, const double* G,
                    const LoadState* st, long long stride, int nload, cudaStream_t stream);
cudaError_t gen_col(int mode, const GridInfo& g, int N, const float2* tw, float2* S, const float* G,
                    const LoadState* st, long long stride, int nload, cudaStream_t stream);

// row pass with rb rows per block (first: no inverse; kinv: the Krylov operator's
// inverse half; Cfld: point-by-point stiffness or null)
cudaError_t gen_row(bool first, bool kinv, const GridInfo& g, const double2* tw, double* E, double2* S,
                    const uint8_t* phase, const double* dC, Control* ctl, LoadState* st, double* partials, double* hist,
                    int nload, int rb, double* Wout, const double* Yaux, const double* Cfld, cudaStream_t stream);
cudaError_t gen_row(bool first, bool kinv, const GridInfo& g, const float2* tw, float* E, float2* S,
                    const uint8_t* phase, const float* dC, Control* ctl, LoadState* st, double* partials, double* hist,
                    int nload, int rb, float* Wout, const float* Yaux, const float* Cfld, cudaStream_t stream);

}  // namespace fh
