// Dynamic shared memory of the kernels.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

namespace fh {

// Lets `kernel` have `bytes` of dynamic shared memory on the current device.  The limit
// belongs to the process and not to a solver or network: it is raised and never lowered,
// so that none on another host thread falls below what its next launch asks for.
// (The most a block can have, for every kernel, would do as well, but leaves kernels of
// small requests less L1 cache: 40 iterations of a 512^2 grid with point-by-point
// stiffness 2.65 ms against 2.61.)
cudaError_t allow_smem(const void* kernel, size_t bytes);

}  // namespace fh
