// Float32 DD(r) counts with one histogram word for two pairs (count32.cuh, D2).
#include <cuda_runtime.h>

#include "count32.cuh"

namespace cf {

// Wherever the (nbins + 2)^2 rows fit beside the rings of 24 warps (up to 23 bins) and
// the default shape runs: faster at every size tried.  Kernel ms with one word per
// pair / for two pairs, 20 log bins, clustered: 1.2M points Rmax 5 0.214 / 0.212, 10
// 0.265 / 0.255, 25 1.123 / 1.052, 50 5.109 / 4.726; 300k Rmax 25 0.165 / 0.159; 30k Rmax 60
// 0.060 / 0.057; 2M uniform Rmax 15 1.041 / 0.987.  The shared-memory atomics and with
// them a seventh of the L1's data path wavefronts fall away.  With 20 warps of 96
// registers (no spills) 1.137 at Rmax 25, with rings half as long 1.125, and with every row
// added to the global counts by itself 0.03 ms more at every size.
bool count32_paired(const PairParams &P, const PairLaunch &L)
{
    const Geom &g = P.g;
    const bool wide = g.periodic && (2 * g.reach_x + 1 > g.ncx || 2 * g.reach_y + 1 > g.ncy);
    return L.chunk != 8 && L.pp == 2 && !L.evals && !L.verify && Lay32<true>::total(P.nbins) <= SMEM_MAX &&
           P.B.n <= (wide ? D2_MAX_POINTS / 9 : D2_MAX_POINTS);
}

cudaError_t launch_count32_paired(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st)
{
    L.smem = Lay32<true>::total(P.nbins);
    return P.lut_lin ? launch_tasks<Count32<16, 2, false, false, 1, true>, 1,
                                    Count32<16, 2, false, false, 1, true, true>>(P, L, sms, st)
                     : launch_tasks<Count32<16, 2, false, false, 0, true>, 1,
                                    Count32<16, 2, false, false, 0, true, true>>(P, L, sms, st);
}

}  // namespace cf
