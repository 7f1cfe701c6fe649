// Launches of the float32 DD(rp, pi) counts (countrp32.cuh).
#include <cuda_runtime.h>

#include "countrp32.cuh"

namespace cf {

namespace {

template <int I, int PP, bool EVALS, bool VERIFY, int MINB>
cudaError_t launch_shape(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st)
{
    constexpr bool SL = I == 16 && PP == 2 && !EVALS;  // the default shape
    return P.lut_lin
               ? launch_tasks<CountRp32<I, PP, EVALS, VERIFY, 1>, MINB, CountRp32<I, PP, EVALS, VERIFY, 1, SL>>(P, L, sms, st)
               : launch_tasks<CountRp32<I, PP, EVALS, VERIFY, 0>, MINB, CountRp32<I, PP, EVALS, VERIFY, 0, SL>>(P, L, sms, st);
}

}  // namespace

int countrp32_smem(int nbins, int npibins)
{
    return align_up(CRP_HIST + (nbins + 2) * (npibins + 1) * 4, 128);
}

cudaError_t launch_countrp32(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st)
{
    L.smem = countrp32_smem(P.nbins, P.npibins);
    if (L.verify)
        return launch_shape<8, 1, true, true, 2>(P, L, sms, st);
    if (L.pp == 2)  // two primaries per lane
        return L.evals ? launch_shape<16, 2, true, false, 2>(P, L, sms, st)
                       : launch_shape<16, 2, false, false, 3>(P, L, sms, st);
    switch (L.chunk) {
    case 16:
        return L.evals ? launch_shape<16, 1, true, false, 2>(P, L, sms, st)
                       : launch_shape<16, 1, false, false, 3>(P, L, sms, st);
    case 32:
        return L.evals ? launch_shape<32, 1, true, false, 2>(P, L, sms, st)
                       : launch_shape<32, 1, false, false, 3>(P, L, sms, st);
    default:
        return L.evals ? launch_shape<8, 1, true, false, 2>(P, L, sms, st)
                       : launch_shape<8, 1, false, false, 3>(P, L, sms, st);
    }
}

}  // namespace cf
