// Pair counting: the kernels of one call (host).
#include <cuda_runtime.h>

#include <mutex>

#include "launch.cuh"
#include "pairs.cuh"

namespace cf {

// Per (kernel, device): the dynamic shared-memory limit set so far (only ever
// raised) and the occupancy per shared-memory size, queried once.
namespace {
struct OccCache {
    const void *kern;
    int dev, smem, occ;
};
struct AttrCache {
    const void *kern;
    int dev, limit;
};
OccCache g_occ[128];
AttrCache g_attr[64];
int g_nocc = 0, g_nattr = 0;
std::mutex g_occ_mu;
}  // namespace

cudaError_t occupancy_of(const void *kern, int smem, int &occ, int threads)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e)
        return e;
    std::lock_guard<std::mutex> lock(g_occ_mu);
    AttrCache *a = nullptr;
    for (int q = 0; q < g_nattr; ++q)
        if (g_attr[q].kern == kern && g_attr[q].dev == dev)
            a = &g_attr[q];
    if (!a || a->limit < smem) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e)
            return e;
        if (!a && g_nattr < 64)
            a = &g_attr[g_nattr++];
        if (a)
            *a = AttrCache{kern, dev, smem};
    }
    for (int q = 0; q < g_nocc; ++q)
        if (g_occ[q].kern == kern && g_occ[q].dev == dev && g_occ[q].smem == smem) {
            occ = g_occ[q].occ;
            return cudaSuccess;
        }
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, smem);
    if (e)
        return e;
    if (g_nocc < 128)
        g_occ[g_nocc++] = OccCache{kern, dev, smem, occ};
    return cudaSuccess;
}

cudaError_t launch_pairs(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st)
{
    L.kernels = 0;
    if (P.n_items <= 0)
        return cudaSuccess;
    const cudaError_t e = launch_neighbours(P, st);
    if (e)
        return e;
    L.kernels = 2;
    if (L.f64)
        return launch_count64(P, L, sms, st);
    if (P.wacc)
        return P.kind == 0 ? launch_sums32(P, L, sms, st) : launch_sumsrp32(P, L, sms, st);
    if (P.kind == 1)
        return launch_countrp32(P, L, sms, st);
    return count32_paired(P, L) ? launch_count32_paired(P, L, sms, st) : launch_count32(P, L, sms, st);
}

}  // namespace cf
