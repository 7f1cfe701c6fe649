// Launches of the binary64 counts (cull64.cuh).
#include <cuda_runtime.h>

#include "cull64.cuh"

namespace cf {

// Shared memory of a binary64 count: [0, 128) free, start table of the
// binning, squared edges and pi edges,
// per warp a ring of secondaries and a queue of pairs, histograms, binary64 sums.
// DD(rp, pi): one histogram copy per warp while three CTAs fit an SM, else fewer
// copies shared by several warps.
int plan_count64(PairParams &P)
{
    const int slots = P.kind == 0 ? P.nbins : P.nbins * P.npibins;
    P.guess_off = 128;
    P.e2_off = P.guess_off + GUESS;
    P.ring_off = align_up(P.e2_off + (P.nbins + 1 + (P.kind == 1 ? P.npibins + 1 : 0)) * 8, 128);
    P.queue_off = P.ring_off + WARPS * RingXYZ::BYTES;
    P.hist_off = align_up(P.queue_off + WARPS * (int)sizeof(CullQueue), 128);
    const int sums = P.wacc ? slots * 16 : 0;
    if (P.kind == 0) {
        P.hcopies = P.wacc ? WARPS : 1;  // of the sums; the counts have a word per lane
        P.acc_off = P.hist_off + P.nbins * 128;
        return align_up(P.acc_off + P.hcopies * sums, 128);
    }
    P.hcopies = 1;
    for (int c = WARPS; c > 1; c >>= 1)
        if (P.hist_off + c * (slots * 4 + sums) <= 75 * 1024) {
            P.hcopies = c;
            break;
        }
    P.acc_off = align_up(P.hist_off + P.hcopies * slots * 4, 16);
    return align_up(P.acc_off + P.hcopies * sums, 128);
}

namespace {

template <int KIND, int EV>
cudaError_t launch_kind(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st)
{
    if (P.wacc)
        return L.evals ? launch_tasks<Cull64<KIND, true, true, EV>, 3>(P, L, sms, st)
                       : launch_tasks<Cull64<KIND, false, true, EV>, 3, Cull64<KIND, false, true, EV, true>>(P, L, sms, st);
    return L.evals ? launch_tasks<Cull64<KIND, true, false, EV>, 3>(P, L, sms, st)
                   : launch_tasks<Cull64<KIND, false, false, EV>, 3, Cull64<KIND, false, false, EV, true>>(P, L, sms, st);
}

}  // namespace

// Two pairs per lane and evaluation hide the latency of the points' loads, but for
// DD(r) of large catalogues, which fills the binary64 pipe with one.  Kernel ms with one
// / two: DD(r) 30k points Rmax 60 0.294 / 0.272; 300k Rmax 25 0.887 / 0.873, Rmax 60 10.19 /
// 10.00; 600k Rmax 15 0.756 / 0.751, Rmax 25 2.847 / 2.847; 1.2M Rmax 25 10.22 / 10.29, Rmax 50
// 80.4 / 80.8; DD(rp, pi) 100k 0.352 / 0.329, 1.2M 21.9 / 21.6; 48 mixed jobs of a batch 44.8 / 43.6.
// A fourth CTA per SM (64 registers) instead: 10.61 at 1.2M, Rmax 25.
cudaError_t launch_count64(const PairParams &P0, PairLaunch &L, int sms, cudaStream_t st)
{
    PairParams P = P0;
    L.smem = plan_count64(P);
    if (P.kind == 1)
        return launch_kind<1, 2>(P, L, sms, st);
    return P.B.n < 600000 ? launch_kind<0, 2>(P, L, sms, st) : launch_kind<0, 1>(P, L, sms, st);
}

}  // namespace cf
