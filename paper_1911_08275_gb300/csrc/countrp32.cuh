// Float32 DD(rp, pi) without sums over chunk tasks (tasks.cuh): the structure of
// count32.cuh with a 2-D histogram.
//
// rp^2 = dx^2 + dy^2 is binned like r^2 (byte table of float32 thresholds with
// 2-component error bands).  pi = |dz| is binned by arithmetic, since its edges
// are uniform: with t' = |dz| npibins / pimax - 1/2 (one fma), adding 1.5 * 2^23
// rounds t' to the nearest integer m, the pi bin, which the sum's low mantissa
// bits hold; m is right unless t' is within rounding of a half-integer, and the
// exact remainder t' - m tells that case apart (beyond pband).  A pair in a flagged
// rp cell or near a pi edge sets a bit of the lane's mask and is settled later,
// 32 at a time, with the main path's increment undone.
//
// Bound: instruction issue, the ALU pipe first (2-D address, clamps, flag bits).
// 1.2M clustered points, 14 x 40 bins, rp 25, pimax 40 (3.8e9 evaluations, GB300):
// 155 instructions per 8-pair step, issue 76 %, kernel 2.59 ms, against 176 per step
// and 3.08 ms when a CTA staged one column pair at a time, searched every window in
// the staged tile and settled flagged pairs where they were found (nearly every
// block of 8 steps has one).  |dz| comes as an operand modifier of scalar
// instructions: as a mask of packed pairs it took one more instruction per pair,
// twice.
#pragma once

#include <type_traits>

#include "tasks.cuh"

namespace cf {

namespace {

constexpr float PI_MAGIC = 12582912.0f;          // 1.5 * 2^23: spacing 1 in [2^23, 2^24)
constexpr uint32_t PI_MAGIC_BITS = 0x4b400000u;  // its bit pattern

// Shared layout: [0, 128) the table's barrier; table; thresholds; squared rp edges;
// per warp a ring of secondaries and a queue of flagged pairs; the histogram,
// (nbins + 2) rows of (npibins + 1) words (row -1 of flagged rp cells, the bins, the
// not-counted row; column npibins not counted), shared by the CTA's warps.
constexpr int CRP_LUT = 128;
constexpr int CRP_THR = CRP_LUT + LUT_MAX;
constexpr int CRP_E2 = CRP_THR + 2 * (NB_MAX + 1) * 4;
constexpr int CRP_RING = (CRP_E2 + (NB_MAX + 1) * 8 + 127) / 128 * 128;
constexpr int CRP_QUEUE = CRP_RING + WARPS * RingXYZ::BYTES;
constexpr int CRP_HIST = CRP_QUEUE + WARPS * (int)sizeof(FlagQueue);

__device__ __forceinline__ void red_shared_add(uint32_t addr, uint32_t v)
{
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(v));
}

// Canonical binary64 rp^2 and |dz| of a pair, image (qx, qy, qz).
__device__ __forceinline__ double canon_rp2(const PairParams &P, int i, int j, int qx, int qy)
{
    const double4_32a a = P.A.pos64[i], b = P.B.pos64[j];
    const double dx = canon_comp(a.x, b.x, (double)qx * P.g.box[0]);
    const double dy = canon_comp(a.y, b.y, (double)qy * P.g.box[1]);
    return __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
}
__device__ __forceinline__ double canon_pi(const PairParams &P, int i, int j, int qz)
{
    return fabs(canon_comp(P.A.pos64[i].z, P.B.pos64[j].z, (double)qz * P.g.box[2]));
}

// The float32 values of one pair, as the sweep computes them.
struct RpPair {
    float rp2;
    uint32_t e;  // table entry: bin, nbins (not counted) or -1 (flagged)
    uint32_t m;  // pi bin, npibins: not counted
    bool edge;   // near a pi edge
};

__device__ __forceinline__ RpPair rp_pair(const PairParams &P, const unsigned char *smem, int i, int j, int qx,
                                          int qy, int qz)
{
    const float *a = P.A.xyz + quad_off((uint32_t)i), *b = P.B.xyz + quad_off((uint32_t)j);
    const float dx = __fsub_rn(b[0], __fsub_rn(a[0], (float)qx * P.boxf[0]));
    const float dy = __fsub_rn(b[4], __fsub_rn(a[4], (float)qy * P.boxf[1]));
    const float dz = __fsub_rn(b[8], __fsub_rn(a[8], (float)qz * P.boxf[2]));
    RpPair r;
    r.rp2 = __fmaf_rn(dy, dy, __fmul_rn(dx, dx));
    const float t = __fmaf_rn(fabsf(dz), P.pscale, -0.5f);
    const float s = __fadd_rn(t, PI_MAGIC);
    r.m = min(__float_as_uint(s) - PI_MAGIC_BITS, (uint32_t)P.npibins);
    r.edge = fabsf(__fsub_rn(t, __fsub_rn(s, PI_MAGIC))) > P.pband;
    const uint32_t c = P.lut_lin ? __float_as_uint(__fmaf_rn(r.rp2, P.lut_scale, LIN_MAGIC)) - LIN_MAGIC_BITS
                                 : (__float_as_uint(r.rp2) >> P.lut_shift) - P.u0;
    r.e = (uint32_t)(int)(signed char)smem[CRP_LUT + min(c, (uint32_t)(P.lut_n - 1))];
    return r;
}

// The pair's true slot k * (npibins + 1) + m, or -1; re: binary64 was needed.
__device__ __forceinline__ int rp_slot(const PairParams &P, const unsigned char *smem, const RpPair &r, int i,
                                       int j, int qx, int qy, int qz, int &re)
{
    int k = r.e < (uint32_t)P.nbins ? (int)r.e : -1, m = r.m < (uint32_t)P.npibins ? (int)r.m : -1;
    if (r.e > (uint32_t)P.nbins) {  // flagged cell
        const int c = thr_count(reinterpret_cast<const float *>(smem + CRP_THR), P.nthr, r.rp2);
        if (c & 1) {
            k = bin_f64(canon_rp2(P, i, j, qx, qy), reinterpret_cast<const double *>(smem + CRP_E2), P.nbins);
            re = 1;
        } else {
            k = (c >= 2 && c <= 2 * P.nbins) ? (c - 2) >> 1 : -1;
        }
    }
    if (k < 0)
        return -1;
    if (r.edge) {
        m = bin_f64(canon_pi(P, i, j, qz), P.P, P.npibins);
        re = 1;
    }
    return m < 0 ? -1 : k * (P.npibins + 1) + m;
}

// Settle the last min(32, qn) flagged pairs of the warp's queue, one per lane: the
// sweep's increment is undone and the pair added to its true slot.  Returns 1 in
// lanes that needed binary64.
__device__ __noinline__ int settle_rp(const PairParams &P, const unsigned char *smem, uint32_t hbase,
                                      const FlagQueue *fq, int qn)
{
    const int lane = threadIdx.x & 31, first = max(0, qn - 32);
    int re = 0;
    __syncwarp();
    if (first + lane < qn) {
        const int i = fq->i[first + lane], j = fq->j[first + lane], im = fq->image[first + lane];
        const int qx = (im & 3) - 1, qy = ((im >> 2) & 3) - 1, qz = ((im >> 4) & 3) - 1;
        const RpPair r = rp_pair(P, smem, i, j, qx, qy, qz);
        if (r.e != (uint32_t)P.nbins) {  // else not counted, and the sweep did not count it
            const int row = P.npibins + 1;
            const int slot = rp_slot(P, smem, r, i, j, qx, qy, qz, re);
            red_shared_add(hbase + (uint32_t)((int)r.e * row + (int)r.m) * 4u, 0xffffffffu);
            if (slot >= 0)
                red_shared_add(hbase + (uint32_t)slot * 4u, 1u);
        }
    }
    __syncwarp();
    return re;
}

// Debug: do the float32 decisions of a pair agree with binary64?  (1 = violation)
__device__ __noinline__ int verify_rp(const PairParams &P, const unsigned char *smem, int i, int j, int image)
{
    const int qx = (image & 3) - 1, qy = ((image >> 2) & 3) - 1, qz = ((image >> 4) & 3) - 1;
    const RpPair r = rp_pair(P, smem, i, j, qx, qy, qz);
    const float *T = reinterpret_cast<const float *>(smem + CRP_THR);
    int c = 0;
    while (c < P.nthr && T[c] <= r.rp2)
        ++c;
    if ((c & 1) || r.edge)
        return 0;  // no claim inside a band
    const int k32 = (c >= 2 && c <= 2 * P.nbins) ? (c - 2) >> 1 : -1;
    const int m32 = r.m < (uint32_t)P.npibins ? (int)r.m : -1;
    const int k64 = bin_f64(canon_rp2(P, i, j, qx, qy), reinterpret_cast<const double *>(smem + CRP_E2), P.nbins);
    const int m64 = bin_f64(canon_pi(P, i, j, qz), P.P, P.npibins);
    const bool c32 = k32 >= 0 && m32 >= 0, c64 = k64 >= 0 && m64 >= 0;
    return c32 != c64 || (c32 && (k32 != k64 || m32 != m64));
}

// LT: table cells linear in rp^2 (1) or on float bits (0).
template <int I, int PP, bool EVALS, bool VERIFY, int LT, bool SL = false>
struct CountRp32 {
    static constexpr int CH = I * PP, JS = 128 / I;
    struct State {
        u64 n_eval, n_rck, n_viol;
        unsigned pending;  // lane pairs since the last flush
        int qn;            // flagged pairs waiting in the warp's queue
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

    static __device__ __forceinline__ bool load(const PairParams &P, unsigned char *smem, State &st,
                                                unsigned phase)
    {
        const bool ok = load_table(P, smem, CRP_LUT, phase, [&]() {
            uint32_t *hist = reinterpret_cast<uint32_t *>(smem + CRP_HIST);
            for (int q = threadIdx.x; q < P.nthr; q += THREADS)
                reinterpret_cast<float *>(smem + CRP_THR)[q] = P.thr[q];
            for (int q = threadIdx.x; q <= P.nbins; q += THREADS)
                reinterpret_cast<double *>(smem + CRP_E2)[q] = P.E2[q];
            for (int q = threadIdx.x; q < (P.nbins + 2) * (P.npibins + 1); q += THREADS)
                hist[q] = 0u;
        });
        st = State{0ull, 0ull, 0ull, 0u, 0};
        return ok;
    }

    template <bool TRI, bool LIN>
    static __device__ __forceinline__ void sweep(const PairParams &P, const unsigned char *smem, State &st,
                                                 uint32_t addr, int j0, int j1, int jlo, int jhi, int jj, int ii,
                                                 const u64 (&XH)[PP], const u64 (&YH)[PP], const u64 (&ZH)[PP],
                                                 int ib, int image, unsigned vmask)
    {
        const u64 MG = pack2(PI_MAGIC, PI_MAGIC), LS = pack2(P.lut_scale, P.lut_scale),
                  LM = pack2(LIN_MAGIC, LIN_MAGIC);
        const float sc = P.pscale, pband = P.pband;
        const uint32_t npi = (uint32_t)P.npibins, rowb = (npi + 1u) * 4u;
        const uint32_t lutb = smem_u32(smem + CRP_LUT), lut_lo = lutb - LIN_MAGIC_BITS,
                       lut_last = (uint32_t)(P.lut_n - 1), lut_hi = lutb + lut_last;
        const uint32_t hbase = smem_u32(smem + CRP_HIST) + rowb;  // row 0 (row -1 before it)
        const uint32_t p0 = addr + 48u * jj;  // this lane's first quad
        const int jf = j0 + 4 * jj;           // its first secondary
        FlagQueue *fq = reinterpret_cast<FlagQueue *>(const_cast<unsigned char *>(smem) + CRP_QUEUE) +
                        (threadIdx.x >> 5);
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
#pragma unroll
                for (int q = 0; q < PP; ++q) {
                    float r[4], t[4], s[4], w[4], g[4];
                    uint32_t cq[4];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const u64 dx = fsub2(h ? vx.y : vx.x, XH[q]), dy = fsub2(h ? vy.y : vy.x, YH[q]);
                        const u64 r2 = ffma2(dy, dy, fmul2(dx, dx));
                        float za, zb;
                        unpack2(fsub2(h ? vz.y : vz.x, ZH[q]), za, zb);
                        // |dz| as an operand modifier of the scalar instructions
                        t[2 * h] = __fmaf_rn(fabsf(za), sc, -0.5f);
                        t[2 * h + 1] = __fmaf_rn(fabsf(zb), sc, -0.5f);
                        const u64 t2 = pack2(t[2 * h], t[2 * h + 1]);
                        const u64 s2 = fadd2(t2, MG);
                        unpack2(r2, r[2 * h], r[2 * h + 1]);
                        unpack2(s2, s[2 * h], s[2 * h + 1]);
                        unpack2(fsub2(t2, fsub2(s2, MG)), w[2 * h], w[2 * h + 1]);
                        if (LIN) {
                            float c[2];
                            unpack2(ffma2(r2, LS, LM), c[0], c[1]);
                            cq[2 * h] = min(__float_as_uint(c[0]) + lut_lo, lut_hi);
                            cq[2 * h + 1] = min(__float_as_uint(c[1]) + lut_lo, lut_hi);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        // sign set: near a pi edge (a NaN of the padding is positive)
                        g[k] = __fsub_rn(pband, fabsf(w[k]));
                        if (!LIN)
                            cq[k] = lutb + min((__float_as_uint(r[k]) >> P.lut_shift) - P.u0, lut_last);
                        if (TRI) {  // pairs with j <= i: not counted, never flagged
                            const bool live = jt + k > ib + q * I + ii;
                            cq[k] = live ? cq[k] : lut_hi;
                            g[k] = live ? g[k] : 1.0f;
                        }
                        if (EVALS)
                            st.n_eval += (((vmask >> q) & 1u) && jt + k >= jlo && jt + k < jhi &&
                                          (!TRI || jt + k > ib + q * I + ii)) ? 1ull : 0ull;
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t e = lds_entry(cq[k]);
                        const uint32_t m = min(__float_as_uint(s[k]) - PI_MAGIC_BITS, npi);
                        red_shared_add(hbase + e * rowb + m * 4u, 1u);
                        // pair (t, k) ends at bit 4 tend - 1 - (4 t + k)
                        fm[q] = push_sign(fm[q], e | __float_as_uint(g[k]));
                        if (VERIFY)
                            if (((vmask >> q) & 1u) && !isnan(r[k]) && (!TRI || jt + k > ib + q * I + ii))
                                st.n_viol += verify_rp(P, smem, ib + q * I + ii, jt + k, image);
                    }
                }
            }
            uint32_t anyf = 0u;
#pragma unroll
            for (int q = 0; q < PP; ++q)
                anyf |= fm[q];
            if (__any_sync(FULL, anyf != 0u)) {
#pragma unroll
                for (int q = 0; q < PP; ++q) {
                    uint32_t m = fm[q];
                    for (unsigned bm; (bm = __ballot_sync(FULL, m != 0u)) != 0u;) {
                        if (m) {
                            const int b = 4 * tend - __ffs(m);  // = 4 t + k
                            const int at = st.qn + __popc(bm & ((1u << (threadIdx.x & 31)) - 1u));
                            fq->i[at] = ib + q * I + ii;
                            fq->j[at] = jf + (int)((pb - p0) / 12u) + (b >> 2) * JS + (b & 3);
                            fq->image[at] = image;
                            m &= m - 1u;
                        }
                        st.qn += __popc(bm);
                        if (st.qn >= 32) {
                            st.n_rck += settle_rp(P, smem, hbase, fq, st.qn);
                            st.qn -= 32;
                        }
                    }
                }
            }
        }
    }

    static __device__ __forceinline__ void task(const PairParams &P, unsigned char *smem, State &st,
                                                unsigned c, unsigned part, unsigned parts)
    {
        const int lane = threadIdx.x & 31, ii = lane % I, jj = lane / I;
        const uint32_t ring = smem_u32(smem + CRP_RING) + (threadIdx.x >> 5) * (uint32_t)RingXYZ::BYTES;
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
                auto go = [&](auto tr, auto li) {
                    sweep<decltype(tr)::value, decltype(li)::value>(P, smem, st, addr, j0, j1, jlo, jhi, jj, ii,
                                                                    XH, YH, ZH, ib, image, C.vmask);
                };
                st.pending += (unsigned)((j1 - j0) / JS + 1) * 4u * PP;
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
                // a warp adds at most 32 to one word per lane pair: keep it below 2^30
                if (st.pending > (1u << 30) / (32u * WARPS) >> FLUSH_SHIFT) {
                    __syncwarp();
                    const int row = P.npibins + 1;
                    uint32_t *hist = reinterpret_cast<uint32_t *>(smem + CRP_HIST) + row;
                    for (int s = lane; s < P.nbins * row; s += 32) {
                        const int b = s / row, m = s - b * row;
                        // signed: an increment flushed earlier may be undone after it
                        const int v = m < P.npibins ? (int)atomicExch(&hist[s], 0u) : 0;
                        if (v)
                            atomicAdd(&P.hist[b * P.npibins + m], (u64)(long long)v);
                    }
                    st.pending = 0;
                }
            });
    }

    static __device__ __forceinline__ void fini(const PairParams &P, unsigned char *smem, State &st)
    {
        const int lane = threadIdx.x & 31, row = P.npibins + 1;
        uint32_t *hist = reinterpret_cast<uint32_t *>(smem + CRP_HIST) + row;
        if (st.qn) {
            st.n_rck += settle_rp(P, smem, smem_u32(hist),
                                  reinterpret_cast<FlagQueue *>(smem + CRP_QUEUE) + (threadIdx.x >> 5), st.qn);
            st.qn = 0;
        }
        __syncthreads();
        for (int s = threadIdx.x; s < P.nbins * P.npibins; s += THREADS) {
            const int b = s / P.npibins, v = (int)hist[b * row + (s - b * P.npibins)];
            if (v)
                atomicAdd(&P.hist[s], (u64)(long long)v);
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
