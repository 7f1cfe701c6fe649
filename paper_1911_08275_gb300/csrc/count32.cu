// Launches of the float32 DD(r) counts (count32.cuh) and the neighbour lists of the
// chunk tasks.
#include <cuda_runtime.h>

#include "count32.cuh"

namespace cf {

namespace {

__global__ void __launch_bounds__(128) k_neighbours(const __grid_constant__ PairParams P)
{
    if (*P.err & ERR_TIMEOUT) {  // the gridding gave up: leave the pair kernel no task
        if (blockIdx.x == 0 && threadIdx.x == 0)
            P.A.cell_start[P.g.ncells] = 0u;
        return;
    }
    neighbours_body(P, (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), threadIdx.x & 31);
}

template <int I, int PP, bool EVALS, bool VERIFY, int MINB>
cudaError_t launch_shape(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st)
{
    constexpr bool SL = I == 16 && PP == 2 && !EVALS;  // the default shape
    return P.lut_lin ? launch_tasks<Count32<I, PP, EVALS, VERIFY, 1>, MINB,
                                    Count32<I, PP, EVALS, VERIFY, 1, false, SL>>(P, L, sms, st)
                     : launch_tasks<Count32<I, PP, EVALS, VERIFY, 0>, MINB,
                                    Count32<I, PP, EVALS, VERIFY, 0, false, SL>>(P, L, sms, st);
}

}  // namespace

int count32_smem(int nbins) { return Lay32<false>::total(nbins); }

cudaError_t launch_neighbours(const PairParams &P, cudaStream_t st)
{
    k_neighbours<<<(P.g.ncols + 3) / 4, 128, 0, st>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_count32(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st)
{
    L.smem = count32_smem(P.nbins);
    if (L.verify)
        return launch_shape<8, 1, true, true, 3>(P, L, sms, st);
    if (L.pp == 4)
        return L.evals ? launch_shape<8, 4, true, false, 2>(P, L, sms, st)
                       : launch_shape<8, 4, false, false, 2>(P, L, sms, st);
    if (L.pp == 2) {
        if (L.chunk == 8)
            return L.evals ? launch_shape<8, 2, true, false, 3>(P, L, sms, st)
                           : launch_shape<8, 2, false, false, 3>(P, L, sms, st);
        return L.evals ? launch_shape<16, 2, true, false, 3>(P, L, sms, st)
                       : launch_shape<16, 2, false, false, 3>(P, L, sms, st);
    }
    switch (L.chunk) {
    case 16:
        return L.evals ? launch_shape<16, 1, true, false, 3>(P, L, sms, st)
                       : launch_shape<16, 1, false, false, 3>(P, L, sms, st);
    case 32:
        return L.evals ? launch_shape<32, 1, true, false, 3>(P, L, sms, st)
                       : launch_shape<32, 1, false, false, 3>(P, L, sms, st);
    default:
        return L.evals ? launch_shape<8, 1, true, false, 3>(P, L, sms, st)
                       : launch_shape<8, 1, false, false, 3>(P, L, sms, st);
    }
}

}  // namespace cf
