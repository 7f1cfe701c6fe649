// Launch helpers of the pair kernels (host).
#pragma once

#include <cuda_runtime.h>

namespace cf {

// CTAs of `threads` threads per SM for a kernel with smem bytes of dynamic shared
// memory; raises the kernel's shared-memory limit when needed, never lowers it (cached).
cudaError_t occupancy_of(const void *kern, int smem, int &occ, int threads = 256);

template <class K>
cudaError_t occupancy(K kern, int smem, int &occ, int threads = 256)
{
    return occupancy_of((const void *)kern, smem, occ, threads);
}

// Parts a split chunk task has (TaskSplit; a part takes every parts-th
// neighbour) for a count of about `chunks` chunks on `warps` warps: 8, more where
// there are fewer than two chunks per warp, so that there are some 16 tasks per
// warp (a chunk of a dense catalogue against all neighbours is a long task).
constexpr int TASK_PARTS = 8;
inline int task_parts(double chunks, double warps, int nstencil)
{
    const double want = 16.0 * warps / (chunks > 1.0 ? chunks : 1.0);
    const int parts = want > TASK_PARTS ? (want < 1024.0 ? (int)want : 1024) : TASK_PARTS;
    return parts < nstencil ? parts : nstencil;
}

}  // namespace cf
