// The cluster kernel's staged FP64 variant (cluster.cuh).
#include "clusterkern.hpp"
#include "cluster.cuh"

namespace fh {

const void* cluster_kernel_staged(double, int nv, int cs) {
  if (cs == 16)
    return nv == 3 ? (const void*)cluster_solve_2d<double, 3, 16, kClusterStaged>
                   : (const void*)cluster_solve_2d<double, 6, 16, kClusterStaged>;
  return nv == 3 ? (const void*)cluster_solve_2d<double, 3, 8, kClusterStaged> : (const void*)cluster_solve_2d<double, 6, 8, kClusterStaged>;
}

CheckUnit check_unit_clusterst64() { return {check_take, check_selftest}; }

}  // namespace fh
