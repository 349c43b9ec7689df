// The cluster kernel's variants (cluster.cuh), compiled in units of their own beside the
// solver, and the choice between them (clusterplan.cpp).
#pragma once

#include "internal.hpp"

namespace fh {

enum ClusterKind {
  kClusterPow2 = 0,     // radices 2, 4 and 8 only, inlined; FP32 lines by single warps
  kClusterGeneral = 1,  // FP32 lines of R1 R2 points by single warps, every radix to 16 (bigfft.cuh)
  kClusterStaged = 2    // radices 2, 3, 4, 5, 7, 8, 11, 13 and direct stages, inlined
};

// kernel and radix schedules of a 2-axis grid (axis 1 contiguous)
struct ClusterChoice {
  int kind = kClusterPow2;
  FftPlan plan0, plan1;
};
bool cluster_choice(int N0, int L, int nv, bool fp32, ClusterChoice* out);

// the kernel for n_v components and clusters of 8 or 16, to be launched with (tasks,
// ntasks, next) on cluster_kernel_threads threads per CTA
const void* cluster_kernel(double, int nv, int cs, int kind);
const void* cluster_kernel(float, int nv, int cs, int kind);
inline int cluster_kernel_threads(bool fp32, int kind) { return fp32 && kind != kClusterStaged ? 512 : 256; }

}  // namespace fh
