// resident.h -- setting up the resident SYNC kernel (kernels_resident.cu), once per swarm.
#pragma once

#include <cuda_runtime.h>

#include "cupso_device.cuh"

namespace cupso {

// Raises the kernel's shared-memory limit; before the swarm's first launch_resident.
cudaError_t prepare_resident(const SwarmDev& s, int fid, int num_sms);

}  // namespace cupso
