// The cluster kernel's variants (cluster.cuh), compiled in one unit per
// precision beside the solver: the kernel for n_v components, cluster size 8 or
// 16 and radix plans of powers of two only (or any), to be launched with
// (tasks, ntasks, next).
#pragma once

#include <cuda_runtime.h>

#include "internal.hpp"
#include "kernels.cuh"

namespace fh {

const void* cluster_kernel(double, int nv, int cs, bool pow2);
const void* cluster_kernel(float, int nv, int cs, bool pow2);

}  // namespace fh
