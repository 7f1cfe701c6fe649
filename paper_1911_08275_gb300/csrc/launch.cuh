// Launch helpers of the pair kernels (host).
#pragma once

#include <cuda_runtime.h>

namespace cf {

// CTAs of THREADS threads per SM for a kernel with smem bytes of dynamic shared
// memory; raises the kernel's shared-memory limit when needed (cached).
cudaError_t occupancy_of(const void *kern, int smem, int &occ);

template <class K>
cudaError_t occupancy(K kern, int smem, int &occ)
{
    return occupancy_of((const void *)kern, smem, occ);
}

// Parts a split chunk task has, at most (TaskSplit); a part takes every
// TASK_PARTS-th neighbour.
constexpr int TASK_PARTS = 8;

}  // namespace cf
