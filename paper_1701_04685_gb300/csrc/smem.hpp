// Dynamic shared memory of the kernels.
#pragma once

#include <cuda_runtime.h>

namespace fh {

// Lets `kernel` have as much dynamic shared memory as a block of the current device can
// (the opt-in limit less the kernel's static part).  The limit belongs to the process and
// not to a solver or network; as every caller sets the same value, none on another host
// thread can lower it between this call and a launch.
cudaError_t allow_smem(const void* kernel);

}  // namespace fh
