// Float32 DD(r) without sums: the hot loop of the paper (Sec. 2.2, Codes 2-4)
// over chunk tasks (tasks.cuh).
//
// Each lane holds PP primaries, each broadcast into both halves of a 64-bit
// register, and evaluates them against four consecutive secondaries (one
// 16-byte load per axis, two packed pairs) with the packed f32x2 instructions.
// The squared distance indexes (clamped, branch-free) a byte table built on the
// host from float32 thresholds lo_k < e_k^2 < hi_k that bracket every squared
// edge by a proven error bound; a safe cell gives the bin row, out-of-range
// distances a dummy row, and every lane adds one to its own column of the CTA's
// shared histogram with a shared-memory atomic (no bank conflicts, no branch).
// A pair in a flagged cell (touching a band) sets a bit of the lane's mask;
// once per 8 steps a warp-uniform test moves the recorded pairs to the warp's
// queue, and whenever 32 wait there they are settled together, one per lane: compared
// with the thresholds, a distance inside a band re-evaluated with the canonical
// binary64 formula, so counts are bit-identical to the binary64 definition.
//
// Bounds, and what was measured (1.2M clustered points, box 420, 20 log bins,
// Rmax 25, 2.3e9 evaluations, GB300): a step of 8 pairs per lane takes 96
// instructions (28 packed float32, 8 each of table byte, atomic, address, clamp
// and flag bit, 3 tile loads) and 28 wavefronts of the L1's data path, which is
// 81 % busy, issue 68 %: the data path binds first.  Kernel 1.127 ms, against
// 1.193 ms for CTAs that staged one column pair at a time in two tile buffers and
// settled flagged pairs where they were found (0.5M pairs in a third of all
// blocks of 8 steps, a whole warp waiting for one lane); without the queue the
// chunk tasks took 1.218 ms, and reading the secondaries through the L1 instead
// of the ring 1.245 ms (four wavefronts per 16-byte load).  Rmax 5 / 10 / 50: 0.282 /
// 0.280 / 5.285 ms before, 0.219 / 0.270 / 5.12 ms so.
//
// Where (nbins + 2)^2 rows fit beside the rings of 24 warps, an atomic takes two pairs
// (D2): the row is that of the pair of entries, and a bin's count is the sum of the
// rows with the bin as either entry.  Four fewer atomics (8 -> 4) and the four
// multiply-adds that join two entries in the place of eight addresses: 24 wavefronts
// a step.  Kernel at Rmax 25 1.052 ms, at Rmax 5 / 10 / 50 0.212 / 0.255 / 4.73 ms.
#pragma once

#include <type_traits>

#include "tasks.cuh"

namespace cf {

namespace {

// Shared layout: [0, 128) the table's barrier; table; thresholds; squared edges;
// per warp a ring of secondaries and a queue of flagged pairs; histogram of
// (nbins + 2) rows of 32 words (row -1 of flagged pairs, the bins, the not-counted
// row), shared by the CTA's warps.
constexpr int C32_LUT = 128;
constexpr int C32_THR = C32_LUT + LUT_MAX;
constexpr int C32_E2 = C32_THR + 2 * (NB_MAX + 1) * 4;
constexpr int C32_RING = (C32_E2 + (NB_MAX + 1) * 8 + 127) / 128 * 128;

// D2: one histogram word for two pairs (a row per pair of entries, (nbins + 2)^2 rows),
// which halves the atomics; a CTA of 24 warps shares it.
template <bool D2>
struct Lay32 {
    static constexpr int NW = D2 ? 24 : WARPS;
    using Ring = RingXYZ;
    static constexpr int QUEUE = C32_RING + NW * Ring::BYTES;
    static constexpr int HIST = QUEUE + NW * (int)sizeof(FlagQueue);
    static __host__ __device__ int words(int nb) { return (D2 ? (nb + 2) * (nb + 2) : nb + 2) * 32; }
    static __host__ __device__ int total(int nb) { return align_up(HIST + words(nb) * 4, 128); }
};

// Secondaries a D2 count may have, so that no word overflows: a warp flushes between
// tasks once it has evaluated 2^30 / 24 pairs per lane, and one task evaluates at most
// 3 (images in z) x 2 (padding) x n pairs per lane, each up to 1.5 additions:
// 24 * 1.5 * 6 * 2^23 + 1.5 * 2^30 < 2^32.  Where the stencil is wider than the grid, a
// column comes up under up to 9 images in x and y.
constexpr long long D2_MAX_POINTS = 1ll << 23;

// What a sweep needs beside the primaries.
struct Sweep {
    uint32_t lutb, hl;  // shared addresses: table, this lane's histogram column (row 0)
    uint32_t u0, lut_last;
    int shift, nthr, nb;
    uint32_t nrow;      // D2: nbins + 2
    // where settled pairs go: row 0 of this lane's column (D2: with a pair that does not
    // count), bytes per row
    template <bool D2>
    __device__ __forceinline__ uint32_t settle_at() const
    {
        return D2 ? hl + (nrow - 2u) * 128u : hl;
    }
    template <bool D2>
    __device__ __forceinline__ uint32_t settle_row() const
    {
        return D2 ? nrow * 128u : 128u;
    }
    float lscale;
    FlagQueue *fq;
    int qn;  // flagged pairs waiting in the warp's queue
};

// Settle the last min(32, qn) flagged pairs of the warp's queue, one per lane (their
// rows are rowb bytes apart from hl): the float32 d2 with the sweep's operations,
// counted against the thresholds; inside a band re-evaluated in binary64.  Each pair goes to its true bin (the sweep has
// put it in row -1, which is never read).  Returns 1 in lanes that re-evaluated.
__device__ __noinline__ int settle(const PairParams &P, const unsigned char *smem, uint32_t hl,
                                   uint32_t rowb, const FlagQueue *fq, int qn)
{
    const int lane = threadIdx.x & 31, first = max(0, qn - 32);
    int row = -1, re = 0;
    __syncwarp();
    if (first + lane < qn) {
        const int i = fq->i[first + lane], j = fq->j[first + lane], m = fq->image[first + lane];
        const int qx = (m & 3) - 1, qy = ((m >> 2) & 3) - 1, qz = ((m >> 4) & 3) - 1;
        const float *a = P.A.xyz + quad_off((uint32_t)i), *b = P.B.xyz + quad_off((uint32_t)j);
        const float dx = __fsub_rn(b[0], __fsub_rn(a[0], (float)qx * P.boxf[0]));
        const float dy = __fsub_rn(b[4], __fsub_rn(a[4], (float)qy * P.boxf[1]));
        const float dz = __fsub_rn(b[8], __fsub_rn(a[8], (float)qz * P.boxf[2]));
        const float d2 = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
        const int c = thr_count(reinterpret_cast<const float *>(smem + C32_THR), P.nthr, d2);
        if (!(c & 1)) {
            row = (c >= 2 && c <= 2 * P.nbins) ? (c - 2) >> 1 : -1;
        } else {
            row = bin_f64(canon_r2(P.A.pos64[i], P.B.pos64[j], (double)qx * P.g.box[0],
                                   (double)qy * P.g.box[1], (double)qz * P.g.box[2]),
                          reinterpret_cast<const double *>(smem + C32_E2), P.nbins);
            re = 1;
        }
    }
    if (row >= 0)
        red_shared1(hl + (uint32_t)row * rowb);
    __syncwarp();
    return re;
}

// Sweep the piece [j0, j1) of a window [jlo, jhi), its secondaries at shared
// address addr.  Lane (ii, jj) holds PP primaries and evaluates them against the
// quad 4 jj .. 4 jj + 3 of each step; a step covers I PP primaries x JS = 128 / I
// secondaries and starts at a multiple of JS, so it never leaves the column
// (columns are padded to 32).  Secondaries outside the window are farther than
// Rmax in z and never counted.  TRI: pairs with j <= i do not count.
template <int I, int PP, bool TRI, bool EVALS, bool VERIFY, bool LIN, bool D2>
__device__ __forceinline__ void sweep(const PairParams &P, const unsigned char *smem, Sweep &S,
                                      uint32_t addr, int j0, int j1, int jlo, int jhi, int jj,
                                      const u64 (&XH)[PP], const u64 (&YH)[PP], const u64 (&ZH)[PP], int ib,
                                      int image, unsigned vmask, u64 &n_eval, u64 &n_rck, u64 &n_viol)
{
    constexpr int JS = 128 / I;
    const float qnan = __int_as_float(0x7fc00000);
    const u64 LS = pack2(S.lscale, S.lscale), LM = pack2(LIN_MAGIC, LIN_MAGIC);
    const uint32_t lut_lo = S.lutb - LIN_MAGIC_BITS, lut_hi = S.lutb + S.lut_last;
    const int ii = (threadIdx.x & 31) % I;
    const uint32_t p0 = addr + 48u * jj;  // this lane's first quad
    const int jf = j0 + 4 * jj;           // its first secondary
    uint32_t p = p0;
    for (int nit = (j1 - j0 + JS - 1) / JS; nit > 0; nit -= 8) {
        const int tend = min(8, nit);
        const uint32_t pb = p, pend = p + (uint32_t)tend * (12u * JS);
        uint32_t fm[PP];
#pragma unroll
        for (int q = 0; q < PP; ++q)
            fm[q] = 0u;
#pragma unroll 1
        for (; p != pend; p += 12 * JS) {
            const int jt = jf + (int)((p - p0) / 12u);  // (TRI and diagnostics only)
            ulonglong2 vx, vy, vz;
            lds128<0>(p, vx);
            lds128<16>(p, vy);
            lds128<32>(p, vz);
            float d[PP][4];
            uint32_t cq[PP][4];
#pragma unroll
            for (int q = 0; q < PP; ++q) {
                u64 dx = fsub2(vx.x, XH[q]), dy = fsub2(vy.x, YH[q]), dz = fsub2(vz.x, ZH[q]);
                const u64 dA = ffma2(dz, dz, ffma2(dy, dy, fmul2(dx, dx)));
                dx = fsub2(vx.y, XH[q]);
                dy = fsub2(vy.y, YH[q]);
                dz = fsub2(vz.y, ZH[q]);
                const u64 dB = ffma2(dz, dz, ffma2(dy, dy, fmul2(dx, dx)));
                unpack2(dA, d[q][0], d[q][1]);
                unpack2(dB, d[q][2], d[q][3]);
                if (LIN) {  // one packed fma gives two cells; the sum is >= 2^23 (NaN larger)
                    float c[4];
                    unpack2(ffma2(dA, LS, LM), c[0], c[1]);
                    unpack2(ffma2(dB, LS, LM), c[2], c[3]);
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        cq[q][r] = min(__float_as_uint(c[r]) + lut_lo, lut_hi);
                } else {
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        cq[q][r] = S.lutb + min((__float_as_uint(d[q][r]) >> S.shift) - S.u0, S.lut_last);
                }
            }
            if (TRI) {
#pragma unroll
                for (int q = 0; q < PP; ++q)
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const bool live = jt + r > ib + q * I + ii;
                        cq[q][r] = live ? cq[q][r] : lut_hi;
                        d[q][r] = live ? d[q][r] : qnan;
                    }
            }
            if (EVALS) {
#pragma unroll
                for (int q = 0; q < PP; ++q)
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        n_eval += (((vmask >> q) & 1u) && jt + r >= jlo && jt + r < jhi &&
                                   (!TRI || jt + r > ib + q * I + ii)) ? 1ull : 0ull;
            }
#pragma unroll
            for (int q = 0; q < PP; ++q) {
                uint32_t e[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    e[r] = lds_entry(cq[q][r]);  // the row: bin, dummy or flagged (-1)
                    if (!D2)
                        red_shared1(S.hl + e[r] * 128u);
                    fm[q] = push_sign(fm[q], e[r]);  // pair (t, r) ends at bit 4 tend - 1 - (4 t + r)
                    if (D2 && (r & 1))
                        red_shared1(S.hl + (e[r - 1] * S.nrow + e[r]) * 128u);
                }
            }
            if (VERIFY) {
                const float *T = reinterpret_cast<const float *>(smem + C32_THR);
                const double *E2 = reinterpret_cast<const double *>(smem + C32_E2);
#pragma unroll
                for (int q = 0; q < PP; ++q)
#pragma unroll
                    for (int r = 0; r < 4; ++r)  // sentinels and padding give NaN
                        if (((vmask >> q) & 1u) && !isnan(d[q][r]))
                            n_viol += verify_pair(d[q][r], T, S.nthr, S.nb, E2, P.A.pos64, P.B.pos64,
                                                  ib + q * I + ii, jt + r,
                                                  (double)((image & 3) - 1) * P.g.box[0],
                                                  (double)(((image >> 2) & 3) - 1) * P.g.box[1],
                                                  (double)(((image >> 4) & 3) - 1) * P.g.box[2]);
            }
        }
        uint32_t anyf = 0u;
#pragma unroll
        for (int q = 0; q < PP; ++q)
            anyf |= fm[q];
        if (__any_sync(FULL, anyf != 0u)) {  // queue the flagged pairs; settle them 32 at a time
#pragma unroll
            for (int q = 0; q < PP; ++q) {
                uint32_t m = fm[q];
                for (unsigned bm; (bm = __ballot_sync(FULL, m != 0u)) != 0u;) {
                    if (m) {
                        const int b = 4 * tend - __ffs(m);  // = 4 t + r
                        const int at = S.qn + __popc(bm & ((1u << (threadIdx.x & 31)) - 1u));
                        S.fq->i[at] = ib + q * I + ii;
                        S.fq->j[at] = jf + (int)((pb - p0) / 12u) + (b >> 2) * JS + (b & 3);
                        S.fq->image[at] = image;
                        m &= m - 1u;
                    }
                    S.qn += __popc(bm);
                    if (S.qn >= 32) {
                        n_rck += settle(P, smem, S.template settle_at<D2>(), S.template settle_row<D2>(), S.fq, S.qn);
                        S.qn -= 32;
                    }
                }
            }
        }
    }
}

// LT: table cells linear in d2 (1) or on float bits (0).
template <int I, int PP, bool EVALS, bool VERIFY, int LT, bool D2 = false, bool SL = false>
struct Count32 {
    using Lay = Lay32<D2>;
    static constexpr int CH = I * PP, NW = Lay::NW, NT = NW * 32;
    struct State {
        Sweep S;
        u64 n_eval, n_rck, n_viol;
        unsigned pending;  // pairs added to this lane's column since the last flush
    };

    static __device__ __forceinline__ bool init(const PairParams &P, unsigned char *smem, State &st)
    {
        if (threadIdx.x == 0) {
            mbar_init(reinterpret_cast<uint64_t *>(smem), 1);
            fence_mbar_init();
        }
        __syncthreads();
        return load(P, smem, st, 0u);
    }

    // The job's tables and an empty histogram; the barrier's phase parity is phase.
    static __device__ __forceinline__ bool load(const PairParams &P, unsigned char *smem, State &st,
                                                unsigned phase)
    {
        uint32_t *hist = reinterpret_cast<uint32_t *>(smem + Lay::HIST);
        const int tid = threadIdx.x, nb = P.nbins;
        const bool ok = load_table(P, smem, C32_LUT, phase, [&]() {
            for (int q = tid; q < P.nthr; q += NT)
                reinterpret_cast<float *>(smem + C32_THR)[q] = P.thr[q];
            for (int q = tid; q <= nb; q += NT)
                reinterpret_cast<double *>(smem + C32_E2)[q] = P.E2[q];
            for (int q = tid; q < Lay::words(nb); q += NT)
                hist[q] = 0u;
        });
        st.n_eval = st.n_rck = st.n_viol = 0ull;
        st.pending = 0u;
        Sweep &S = st.S;
        S.lutb = smem_u32(smem + C32_LUT);
        S.nrow = (uint32_t)nb + 2u;
        S.hl = smem_u32(hist + (D2 ? nb + 3 : 1) * 32 + (tid & 31));  // row 0 (row -1 before it)
        S.u0 = P.u0;
        S.lut_last = (uint32_t)(P.lut_n - 1);
        S.shift = P.lut_shift;
        S.nthr = P.nthr;
        S.nb = nb;
        S.lscale = P.lut_scale;
        S.fq = reinterpret_cast<FlagQueue *>(smem + Lay::QUEUE) + (tid >> 5);
        S.qn = 0;
        return ok;
    }

    static __device__ __forceinline__ void task(const PairParams &P, unsigned char *smem, State &st,
                                                unsigned c, unsigned part, unsigned parts)
    {
        const int lane = threadIdx.x & 31, ii = lane % I, jj = lane / I;
        const uint32_t ring = smem_u32(smem + C32_RING) + (threadIdx.x >> 5) * (uint32_t)Lay::Ring::BYTES;
        const int ib = (int)(c * CH);
        Chunk<I, PP> C;
        if (!C.load(P, ib, ii))
            return;
        u64 XH[PP], YH[PP], ZH[PP];
        int image = 0;
        for_windows<128 / I, typename Lay::Ring, SL>(
            P, C.col, ib, C.zlo, C.zhi, (int)part, (int)parts, lane, ring,
            [&](int k, int code) { image = C.shift(P, k, code, XH, YH, ZH); },
            [&](uint32_t addr, int j0, int j1, int jlo, int jhi, bool tri) {
                auto go = [&](auto tr, auto li) {
                    sweep<I, PP, decltype(tr)::value, EVALS, VERIFY, decltype(li)::value, D2>(
                        P, smem, st.S, addr, j0, j1, jlo, jhi, jj, XH, YH, ZH, ib, image, C.vmask, st.n_eval,
                        st.n_rck, st.n_viol);
                };
                st.pending += (unsigned)((j1 - j0) / (128 / I) + 1) * 4u * PP;
                if (LT == 1) {
                    if (tri)
                        go(std::true_type{}, std::true_type{});
                    else
                        go(std::false_type{}, std::true_type{});
                } else {
                    if (tri)
                        go(std::true_type{}, std::false_type{});
                    else
                        go(std::false_type{}, std::false_type{});
                }
                if (!D2 && st.pending > (1u << 30) / NW >> FLUSH_SHIFT) {  // keep every shared u32 count far from overflow
                    __syncwarp();
                    warp_flush_shared(reinterpret_cast<uint32_t *>(smem + Lay::HIST) + 32, P.nbins, P.hist,
                                      lane);
                    st.pending = 0;
                }
            });
        if (D2 && st.pending > (1u << 30) / NW >> FLUSH_SHIFT) {
            __syncwarp();
            flush(P, smem, lane, 1, 0);
            st.pending = 0;
        }
    }

    // Rows w0, w0 + step, ... to the global counts, each word taken by one exchange (other
    // warps may be adding).  D2: a row's pairs belong to two bins.
    static __device__ __noinline__ void flush(const PairParams &P, unsigned char *smem, int lane, int step, int w0)
    {
        uint32_t *hist = reinterpret_cast<uint32_t *>(smem + Lay::HIST);
        const int nb = P.nbins, nr = nb + 2;
        for (int r = w0; r < (D2 ? nr * nr : nr); r += step) {
            const int b1 = (D2 ? r % nr : r) - 1, b0 = D2 ? r / nr - 1 : -1;
            const bool in1 = b1 >= 0 && b1 < nb, in0 = b0 >= 0 && b0 < nb;
            if (!in0 && !in1)
                continue;
            const u64 v = warp_sum_u64(atomicExch(&hist[r * 32 + lane], 0u));
            if (lane == 0 && v) {
                if (in1)
                    atomicAdd(&P.hist[b1], v);
                if (in0)
                    atomicAdd(&P.hist[b0], v);
            }
        }
    }

    static __device__ __forceinline__ void fini(const PairParams &P, unsigned char *smem, State &st)
    {
        const int lane = threadIdx.x & 31;
        if (st.S.qn) {
            st.n_rck += settle(P, smem, st.S.template settle_at<D2>(), st.S.template settle_row<D2>(), st.S.fq, st.S.qn);
            st.S.qn = 0;
        }
        __syncthreads();
        if (D2) {  // a warp per bin: the rows with the bin as either entry
            const uint32_t *hist = reinterpret_cast<const uint32_t *>(smem + Lay::HIST);
            const int nr = P.nbins + 2;
            for (int b = threadIdx.x >> 5; b < P.nbins; b += NW) {
                u64 v = 0;
                for (int c = 0; c < nr; ++c)
                    v += (u64)hist[((b + 1) * nr + c) * 32 + lane] + hist[(c * nr + b + 1) * 32 + lane];
                v = warp_sum_u64(v);
                if (lane == 0 && v)
                    atomicAdd(&P.hist[b], v);
            }
        } else {
            flush(P, smem, lane, NW, threadIdx.x >> 5);
        }
        const u64 n_rck = warp_sum_u64(st.n_rck);
        if (lane == 0 && n_rck)
            atomicAdd(&P.diag[2], n_rck);
        if (EVALS || VERIFY) {
            const u64 n_eval = warp_sum_u64(st.n_eval), n_viol = warp_sum_u64(st.n_viol);
            if (lane == 0) {
                if (n_eval)
                    atomicAdd(&P.diag[1], n_eval);
                if (n_viol)
                    atomicAdd(&P.diag[3], n_viol);
            }
        }
    }
};

}  // namespace

}  // namespace cf
