// Binary64 counts (CF_MODE_FP64): every pair that counts is evaluated with the
// canonical binary64 formula and binned by exact compares of squared edges.
//
// This GPU has two binary64 lanes per SM, so a binary64 instruction holds its
// pipe for 16 cycles, and the windows of a chunk hold three pairs beyond Rmax for
// every one within.  The sweep therefore only discards, with packed float32: a
// pair is dropped when its float32 distance proves it out of reach (the bound
// that brackets the last edge in the float32 tables, build_thresholds; pimax plus
// the window slack for |dz|), as the bounding boxes and z windows drop it.  The
// others are queued per warp, and 32 or 64 at a time are evaluated, one or two per lane,
// so the binary64 pipe works on full warps of pairs that count (all but those in
// the thin shell of the bound and below the first edge).
//
// Bound: the binary64 pipe, 8 instructions per counted pair (DD(rp, pi): 6).  1.2M
// clustered points, kernel ms at Rmax 10 / 25 / 50 (GB300): 5.78 / 40.8 / 198 when every
// pair of the windows was evaluated in binary64, 0.91 / 10.2 / 80.4 now (0.65e9 pairs
// within reach at Rmax 25, 5.1e9 at 50: the pipe alone takes 8.9 and 69.5 ms);
// DD(rp, pi) 14 x 40, pimax 40: 56.8 -> 21.6 (15.8).  Tests of the periodic shift as
// doubles had cost 11.5 instead of 10.3 ms at Rmax 25, a binary search of the
// edges instead of the start table 24.3 instead of 22.0 ms for DD(rp, pi).
#pragma once

#include "tasks.cuh"

namespace cf {

namespace {

// The image of a queued pair when no coordinate is shifted.
constexpr int IMAGE_NONE = 1 | (1 << 2) | (1 << 4);

// Start table of the exact binning: entry q counts the squared edges at or below
// the smallest value whose float32 truncation has the leading bits q (sign 0,
// exponent, three mantissa bits), so a value's bin is found by moving up from there.
constexpr int GUESS = 2048;

// Leading bits of the float32 truncation of v >= 0 (0 below the float32 range).
__device__ __forceinline__ int lead_bits(double v)
{
    const int h = __double2hiint(v) - (896 << 20);  // rebias the exponent: 1023 - 127
    return min(max(h, 0) >> 17, GUESS - 1);
}

// Bin of a binary64 squared separation: k with E2[k] <= v < E2[k + 1], else -1.
__device__ __forceinline__ int bin_guess(double v, const double *E2, const unsigned char *guess, int nb)
{
    const long long u = __double_as_longlong(v);  // non-negative doubles order like their bits
    const long long *e = reinterpret_cast<const long long *>(E2);
    int c = guess[lead_bits(v)];
    while (c <= nb && e[c] <= u)
        ++c;
    return c <= nb ? c - 1 : -1;
}

// Bin of |dz| among the pi edges Pe[0 .. n], from its place on a uniform scale.
__device__ __forceinline__ int bin_pi(double v, const double *Pe, int n, float scale)
{
    const long long u = __double_as_longlong(v);
    const long long *e = reinterpret_cast<const long long *>(Pe);
    if (u >= e[n])
        return -1;
    const float f = __int_as_float(max(__double2hiint(v) - (896 << 20), 0) << 3);  // 20 bits of v
    int p = min((int)(f * scale), n - 1);
    while (p > 0 && e[p] > u)
        --p;
    while (e[p + 1] <= u)
        ++p;
    return p;
}

// Pairs waiting to be evaluated (one queue per warp; at most 32 EV - 1 <= 63 wait when up
// to 32 more are pushed).
struct CullQueue {
    int i[96], j[96], image[96];
};

// Evaluate the n <= 32 EV pairs from entry `first` of the warp's queue, EV per lane,
// their points requested together.
template <int KIND, bool WACC, int EV>
__device__ __noinline__ void eval64(const PairParams &P, unsigned char *smem, const CullQueue *fq,
                                    int first, int n, uint32_t hist, double *acc)
{
    const int lane = threadIdx.x & 31, nb = P.nbins, npi = P.npibins;
    const double *E2 = reinterpret_cast<const double *>(smem + P.e2_off), *Pe = E2 + nb + 1;
    const unsigned char *guess = smem + P.guess_off;
    __syncwarp();
    double4_32a a[EV], b[EV];
#pragma unroll
    for (int u = 0; u < EV; ++u) {  // (entry `first` in the place of those beyond n)
        const int e = first + (lane + 32 * u < n ? lane + 32 * u : 0);
        a[u] = P.A.pos64[fq->i[e]];
        b[u] = P.B.pos64[fq->j[e]];
    }
#pragma unroll
    for (int u = 0; u < EV; ++u) {
        if (lane + 32 * u >= n)
            continue;
        const int m = fq->image[first + lane + 32 * u];
        // canonical differences: fl(x_j - x_i), then fl(+ S) where the image is shifted
        // (integer tests: a compare of doubles would hold the binary64 pipe too)
        double dx = __dsub_rn(b[u].x, a[u].x), dy = __dsub_rn(b[u].y, a[u].y), dz = __dsub_rn(b[u].z, a[u].z);
        if (m != IMAGE_NONE) {
            const int qx = (m & 3) - 1, qy = ((m >> 2) & 3) - 1, qz = ((m >> 4) & 3) - 1;
            if (qx)
                dx = __dadd_rn(dx, qx > 0 ? P.g.box[0] : -P.g.box[0]);
            if (qy)
                dy = __dadd_rn(dy, qy > 0 ? P.g.box[1] : -P.g.box[1]);
            if (qz)
                dz = __dadd_rn(dz, qz > 0 ? P.g.box[2] : -P.g.box[2]);
        }
        double s2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
        if (KIND == 0)
            s2 = __dadd_rn(s2, __dmul_rn(dz, dz));
        int k = bin_guess(s2, E2, guess, nb);
        if (KIND == 1 && k >= 0) {
            const int p = bin_pi(fabs(dz), Pe, npi, P.pscale);
            k = p >= 0 ? k * npi + p : -1;
        }
        if (k >= 0) {
            red_shared1(hist + (uint32_t)k * (KIND == 0 ? 128u : 4u));
            if (WACC) {  // Code 1's weight: the exact product and square root
                const double pw = P.weighted ? __dmul_rn(a[u].w, b[u].w) : 1.0;
                atomicAdd(acc + 2 * k, pw);
                if (P.want_r)
                    atomicAdd(acc + 2 * k + 1, __dmul_rn(__dsqrt_rn(s2), pw));
            }
        }
    }
    __syncwarp();
}

// KIND 0: DD(r), a histogram of nbins rows of 32 words (a word per lane) shared by
// the CTA's warps.  KIND 1: DD(rp, pi), P.hcopies copies of nbins * npibins words.
// WACC: binary64 sums [copy][slot][w, r w] (DD(r): one copy per warp).  EV: pairs per
// lane of one evaluation.
template <int KIND, bool EVALS, bool WACC, int EV, bool SL = false>
struct Cull64 {
    static constexpr int I = 16, PP = 2, CH = I * PP, JS = 128 / I;
    struct State {
        u64 n_eval;
        unsigned pending;  // evaluations by this warp since its copy's last flush
        int qn;            // pairs waiting in the warp's queue
    };

    static __device__ __forceinline__ int slots(const PairParams &P)
    {
        return KIND == 0 ? P.nbins : P.nbins * P.npibins;
    }

    static __device__ __forceinline__ bool load(const PairParams &P, unsigned char *smem, State &st, unsigned)
    {
        return init(P, smem, st);
    }

    static __device__ __forceinline__ bool init(const PairParams &P, unsigned char *smem, State &st)
    {
        double *E2 = reinterpret_cast<double *>(smem + P.e2_off), *Pe = E2 + P.nbins + 1;
        uint32_t *hist = reinterpret_cast<uint32_t *>(smem + P.hist_off);
        double *acc = reinterpret_cast<double *>(smem + P.acc_off);
        const int words = KIND == 0 ? P.nbins * 32 : P.hcopies * slots(P);
        for (int q = threadIdx.x; q <= P.nbins; q += THREADS)
            E2[q] = P.E2[q];
        if (KIND == 1)
            for (int q = threadIdx.x; q <= P.npibins; q += THREADS)
                Pe[q] = P.P[q];
        for (int q = threadIdx.x; q < words; q += THREADS)
            hist[q] = 0u;
        if (WACC)
            for (int q = threadIdx.x; q < P.hcopies * slots(P) * 2; q += THREADS)
                acc[q] = 0.0;
        __syncthreads();
        for (int q = threadIdx.x; q < GUESS; q += THREADS) {
            // smallest value of the cell (cell 0 also holds what lies below the float32
            // range); integer compares, as the binary64 pipe is narrow
            const long long lo = q ? ((long long)((q << 17) + (896 << 20))) << 32 : 0ll;
            int c = 0, hi = P.nbins + 1;
            while (c < hi) {
                const int mid = (c + hi) >> 1;
                if (reinterpret_cast<const long long *>(E2)[mid] <= lo)
                    c = mid + 1;
                else
                    hi = mid;
            }
            smem[P.guess_off + q] = (unsigned char)c;
        }
        st = State{0ull, 0u, 0};
        __syncthreads();
        return true;
    }

    // Evaluate what the warp's queue holds beyond `keep` pairs (keep = 32 EV - 1:
    // full warps only; 0: everything).
    static __device__ __forceinline__ void drain(const PairParams &P, unsigned char *smem, State &st,
                                                 const CullQueue *fq, int keep)
    {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, copy = warp % P.hcopies;
        uint32_t *hw = reinterpret_cast<uint32_t *>(smem + P.hist_off) + (KIND == 0 ? lane : copy * slots(P));
        double *acc = reinterpret_cast<double *>(smem + P.acc_off) + (long long)copy * slots(P) * 2;
        while (st.qn > keep) {
            const int n = min(32 * EV, st.qn);
            st.qn -= n;
            eval64<KIND, WACC, EV>(P, smem, fq, st.qn, n, smem_u32(hw), acc);
            st.pending += EV;
        }
    }

    static __device__ __forceinline__ void task(const PairParams &P, unsigned char *smem, State &st,
                                                unsigned c, unsigned part, unsigned parts)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, ii = lane % I, jj = lane / I;
        CullQueue *fq = reinterpret_cast<CullQueue *>(smem + P.queue_off) + warp;
        const uint32_t ring = smem_u32(smem + P.ring_off) + (uint32_t)warp * RingXYZ::BYTES;
        const int ib = (int)(c * CH);
        Chunk<I, PP> C;
        if (!C.load(P, ib, ii))
            return;
        u64 XH[PP], YH[PP], ZH[PP];
        int image = 0;
        for_windows<JS, RingXYZ, SL>(
            P, C.col, ib, C.zlo, C.zhi, (int)part, (int)parts, lane, ring,
            [&](int k, int code) { image = C.shift(P, k, code, XH, YH, ZH); },
            [&](uint32_t addr, int j0, int j1, int jlo, int jhi, bool tri) {
                cull_piece<KIND, I, PP, EVALS>(P, fq, st.qn, st.n_eval, addr, j0, j1, jlo, jhi, tri, jj, ii, XH,
                                               YH, ZH, ib, image, C.vmask, [&]() { drain(P, smem, st, fq, 32 * EV - 1); });
                flush(P, smem, st);
            });
        // entries name their points, so a partly filled queue waits for the next task
    }

    // Keep every shared u32 count far from overflow.
    static __device__ __forceinline__ void flush(const PairParams &P, unsigned char *smem, State &st)
    {
        if (st.pending < (KIND == 0 ? 1u << 27 : 1u << 22) >> FLUSH_SHIFT)
            return;
        const int lane = threadIdx.x & 31;
        uint32_t *hist = reinterpret_cast<uint32_t *>(smem + P.hist_off);
        __syncwarp();
        if (KIND == 0) {
            warp_flush_shared(hist, P.nbins, P.hist, lane);
        } else {
            uint32_t *hc = hist + ((threadIdx.x >> 5) % P.hcopies) * slots(P);
            for (int s = lane; s < slots(P); s += 32) {
                const uint32_t v = atomicExch(&hc[s], 0u);
                if (v)
                    atomicAdd(&P.hist[s], (u64)v);
            }
        }
        st.pending = 0;
    }

    static __device__ __forceinline__ void fini(const PairParams &P, unsigned char *smem, State &st)
    {
        const int tid = threadIdx.x, lane = tid & 31, n = slots(P);
        drain(P, smem, st, reinterpret_cast<CullQueue *>(smem + P.queue_off) + (tid >> 5), 0);
        __syncthreads();
        const uint32_t *hist = reinterpret_cast<const uint32_t *>(smem + P.hist_off);
        const double *acc = reinterpret_cast<const double *>(smem + P.acc_off);
        if (KIND == 0) {
            for (int b = tid >> 5; b < n; b += WARPS) {
                const u64 v = warp_sum_u64(hist[b * 32 + lane]);
                if (lane == 0 && v)
                    atomicAdd(&P.hist[b], v);
            }
        } else {
            for (int s = tid; s < n; s += THREADS) {
                u64 v = 0;
                for (int c = 0; c < P.hcopies; ++c)
                    v += hist[c * n + s];
                if (v)
                    atomicAdd(&P.hist[s], v);
            }
        }
        if (WACC)
            for (int s = tid; s < n; s += THREADS) {
                double ws = 0.0, rs = 0.0;
                for (int c = 0; c < P.hcopies; ++c) {
                    ws += acc[2 * (c * n + s)];
                    rs += acc[2 * (c * n + s) + 1];
                }
                if (ws != 0.0 || rs != 0.0) {
                    atomicAdd(&P.wsum[s], ws);
                    if (P.want_r)
                        atomicAdd(&P.rsum[s], rs);
                }
            }
        if (EVALS) {
            const u64 v = warp_sum_u64(st.n_eval);
            if (lane == 0 && v)
                atomicAdd(&P.diag[1], v);
        }
    }
};

}  // namespace

}  // namespace cf
