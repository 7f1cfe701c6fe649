// Launches of the float32 DD(rp, pi) sums (sumsrp32.cuh).
#include <cuda_runtime.h>

#include "sumsrp32.cuh"

namespace cf {

namespace {
template <bool W, bool RV, bool RL>
cudaError_t launch_kind(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st)
{
    L.smem = align_up(SumsRp32<2, W, RV, RL, false, true>::SLOTS + P.nbins * P.npibins * 20, 128);
    if (L.evals)
        return P.lut_lin ? launch_tasks<SumsRp32<2, W, RV, RL, true, true>, 3>(P, L, sms, st)
                         : launch_tasks<SumsRp32<2, W, RV, RL, true, false>, 3>(P, L, sms, st);
    return P.lut_lin
               ? launch_tasks<SumsRp32<2, W, RV, RL, false, true>, 3, SumsRp32<2, W, RV, RL, false, true, true>>(P, L, sms, st)
               : launch_tasks<SumsRp32<2, W, RV, RL, false, false>, 3, SumsRp32<2, W, RV, RL, false, false, true>>(P, L, sms, st);
}

}  // namespace

cudaError_t launch_sumsrp32(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st)
{
    if (P.want_r && P.rlo)  // rp from residual-corrected squared separations
        return P.weighted ? launch_kind<true, true, true>(P, L, sms, st)
                          : launch_kind<false, true, true>(P, L, sms, st);
    if (P.weighted && P.want_r)
        return launch_kind<true, true, false>(P, L, sms, st);
    return P.weighted ? launch_kind<true, false, false>(P, L, sms, st)
                      : launch_kind<false, true, false>(P, L, sms, st);
}

}  // namespace cf
