// Launch helpers of the pair kernels (host).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>

#include "cf_internal.cuh"

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

// Slices every window is cut into besides, where even one neighbour per part leaves fewer
// than 8 tasks per warp (some primaries against many secondaries: a window then has a
// column's full depth): slices of at least SLICE_MIN of its about `window` secondaries.
// Kernel ms with whole windows and with 3 / 5 / 8 / 16 tasks per warp: 1,000 x 2M points Rmax
// 60 4.51, 0.36 / 0.33 / 0.33 / 0.36, binary64 17.7, 1.40 / 1.06 / 0.86 / 0.77; 8,000 x 3M Rmax
// 30 1.23, 0.57 / 0.50 / 0.49 / 0.49; 30,000 auto Rmax 205 0.257, 0.259 / 0.260 / 0.258 /
// 0.281.  Kernels of their own: in the set-up of the others slices cost DD(r) 1 % and
// DD(rp, pi) 3 % (registers).
constexpr double SLICE_MIN = 256.0;
inline int task_slices(double chunks, double warps, int nstencil, double window)
{
    const double want = std::min(8.0 * warps / std::max(chunks, 1.0), 1024.0);
    return (int)std::max(1.0, std::min(want / nstencil, window / SLICE_MIN));
}

// Secondaries in a window of a chunk of ch primaries, were the points spread evenly.
inline double window_points(const PairParams &P, int ch)
{
    const double span = P.g.extent[2] * std::min(1.0, (double)ch * P.g.ncols / std::max((double)P.A.n, 1.0));
    const double reach = std::min(P.g.extent[2], 2.0 * P.rz + span);
    return (double)P.B.n / P.g.ncols * (P.g.extent[2] > 0.0 ? reach / P.g.extent[2] : 1.0);
}

}  // namespace cf
