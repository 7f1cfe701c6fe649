// Launches of the float32 DD(r) sums (sums32.cuh).
#include <cuda_runtime.h>

#include "sums32.cuh"

namespace cf {

namespace {

template <int PP, bool W, bool RV, bool RL>
cudaError_t launch_kind(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st)
{
    L.smem = SumLayout<W, RV, RL>::total(P.nbins);
    if (L.evals)
        return P.lut_lin ? launch_tasks<Sums32<PP, W, RV, RL, true, 1>, 2>(P, L, sms, st)
                         : launch_tasks<Sums32<PP, W, RV, RL, true, 0>, 2>(P, L, sms, st);
    return P.lut_lin
               ? launch_tasks<Sums32<PP, W, RV, RL, false, 1>, 2, Sums32<PP, W, RV, RL, false, 1, true>>(P, L, sms, st)
               : launch_tasks<Sums32<PP, W, RV, RL, false, 0>, 2, Sums32<PP, W, RV, RL, false, 0, true>>(P, L, sms, st);
}

}  // namespace

cudaError_t launch_sums32(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st)
{
    if (P.want_r && P.rlo)  // r from residual-corrected squared distances
        return P.weighted ? launch_kind<2, true, true, true>(P, L, sms, st)
                          : launch_kind<2, false, true, true>(P, L, sms, st);
    if (P.weighted && P.want_r)
        return launch_kind<2, true, true, false>(P, L, sms, st);
    return P.weighted ? launch_kind<2, true, false, false>(P, L, sms, st)
                      : launch_kind<2, false, true, false>(P, L, sms, st);
}

}  // namespace cf
