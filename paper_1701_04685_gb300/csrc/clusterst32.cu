// The cluster kernel's staged FP32 variant (cluster.cuh).
#include "clusterkern.hpp"
#include "cluster.cuh"

namespace fh {

const void* cluster_kernel_staged(float, int nv, int cs) {
  if (cs == 16)
    return nv == 3 ? (const void*)cluster_solve_2d<float, 3, 16, kClusterStaged>
                   : (const void*)cluster_solve_2d<float, 6, 16, kClusterStaged>;
  return nv == 3 ? (const void*)cluster_solve_2d<float, 3, 8, kClusterStaged> : (const void*)cluster_solve_2d<float, 6, 8, kClusterStaged>;
}

CheckUnit check_unit_clusterst32() { return {check_take, check_selftest}; }

}  // namespace fh
