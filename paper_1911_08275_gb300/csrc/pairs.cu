// Pair counting: the kernels of one call (host).
#include <cuda_runtime.h>

#include <mutex>

#include "launch.cuh"
#include "pairs.cuh"

namespace cf {

// Per kernel and device: the dynamic shared-memory limit known to be set, and the
// occupancy per shared-memory size.  The limit is only ever raised, also when the table
// is full and it has to be asked for: a planned batch launches with the size it was
// planned for, whatever other calls have needed since.  (Fixed tables: the calls that
// allocate nothing come through here too.)
namespace {
struct KernelKey {
    const void *kern;
    int dev;
    bool operator==(const KernelKey &o) const { return kern == o.kern && dev == o.dev; }
};
struct LimitEntry {
    KernelKey key;
    int limit;
};
struct OccEntry {
    KernelKey key;
    int smem, occ;
};
LimitEntry g_limit[256];
OccEntry g_occ[256];
int g_nlimit = 0, g_nocc = 0;
std::mutex g_occ_mu;

cudaError_t raise_limit(const KernelKey &key, int smem)
{
    for (int q = 0; q < g_nlimit; ++q)
        if (g_limit[q].key == key && g_limit[q].limit >= smem)
            return cudaSuccess;
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, key.kern);
    if (!e && a.maxDynamicSharedSizeBytes < smem)
        e = cudaFuncSetAttribute(key.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e)
        return e;
    const int limit = smem > a.maxDynamicSharedSizeBytes ? smem : a.maxDynamicSharedSizeBytes;
    for (int q = 0; q < g_nlimit; ++q)
        if (g_limit[q].key == key) {
            g_limit[q].limit = limit;
            return cudaSuccess;
        }
    if (g_nlimit < 256)
        g_limit[g_nlimit++] = LimitEntry{key, limit};
    return cudaSuccess;
}
}  // namespace

cudaError_t occupancy_of(const void *kern, int smem, int &occ, int threads)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e)
        return e;
    const KernelKey key{kern, dev};
    std::lock_guard<std::mutex> lock(g_occ_mu);
    if ((e = raise_limit(key, smem)))
        return e;
    for (int q = 0; q < g_nocc; ++q)
        if (g_occ[q].key == key && g_occ[q].smem == smem) {
            occ = g_occ[q].occ;
            return cudaSuccess;
        }
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, smem);
    if (!e && g_nocc < 256)
        g_occ[g_nocc++] = OccEntry{key, smem, occ};
    return e;
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
