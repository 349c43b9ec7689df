// The cluster kernel's FP32 variants for powers of two and for general lengths
// (cluster.cuh).
#include "clusterkern.hpp"
#include "cluster.cuh"

namespace fh {

const void* cluster_kernel_staged(float, int nv, int cs);   // a unit of its own, to compile beside this one

template <int NV, int CS>
static const void* variant(int kind) {
  return kind == kClusterPow2 ? (const void*)cluster_solve_2d<float, NV, CS, kClusterPow2>
                              : (const void*)cluster_solve_2d<float, NV, CS, kClusterGeneral>;
}

const void* cluster_kernel(float, int nv, int cs, int kind) {
  if (kind == kClusterStaged) return cluster_kernel_staged(float(0), nv, cs);
  if (cs == 16) return nv == 3 ? variant<3, 16>(kind) : variant<6, 16>(kind);
  return nv == 3 ? variant<3, 8>(kind) : variant<6, 8>(kind);
}

CheckUnit check_unit_cluster32() { return {check_take, check_selftest}; }

}  // namespace fh
