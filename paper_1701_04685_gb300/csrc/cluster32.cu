// The cluster kernel's FP32 variants (cluster.cuh).
#include "clusterkern.hpp"
#include "cluster.cuh"

namespace fh {

template <int NV>
static const void* variant(int cs, bool pow2) {
  if (cs == 16)
    return pow2 ? (const void*)cluster_solve_2d<float, NV, 16, true> : (const void*)cluster_solve_2d<float, NV, 16, false>;
  return pow2 ? (const void*)cluster_solve_2d<float, NV, 8, true> : (const void*)cluster_solve_2d<float, NV, 8, false>;
}

const void* cluster_kernel(float, int nv, int cs, bool pow2) { return nv == 3 ? variant<3>(cs, pow2) : variant<6>(cs, pow2); }

CheckUnit check_unit_cluster32() { return {check_take, check_selftest}; }

}  // namespace fh
