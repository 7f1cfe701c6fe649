// Float32 DD(rp, pi) with pair weights and / or mean separations over chunk tasks:
// the sweep of countrp32.cuh; a pair that counts adds its terms on the spot, a flagged
// one is queued and settled with its terms, 32 at a time.
//
// Sums: a term v (float32: w = fl(w_i w_j), rp w) is added as the integer v * scale,
// scale a power of two (of its rp bin for rp w) with terms at most 2^41 in size: a
// 32-bit atomic on the low word returns whether it carried, a second one adds the
// high part.  A term of at least 2^23 units is an integer exactly (24 bits), so the
// sums are exact; a smaller one (2^-17 of the largest or less), or one that is not
// finite, is added in binary64 to the global sum.  Shared binary64 atomics, which
// this replaces, are loops of compare-and-swap.
//
// Bound: the shared-memory atomics and the divergent adds.  150k x 300k points, open
// box, 14 x 40 bins, weights and mean rp (8.6e7 pairs counted): 5.13 -> 0.90 ms;
// 1.2M points auto: 79 -> 10.1 ms.  Queueing every pair within reach and evaluating
// full warps from global memory took 2.09 ms: fourteen gathers of 32 addresses.
// Two primaries per lane at three CTAs per SM (200 bytes of spill stores and 300 of loads per
// thread): 0.90 ms, at two CTAs 1.03, one primary per lane 1.03 and 1.16.
#pragma once

#include "countrp32.cuh"
#include "sums32.cuh"

namespace cf {

namespace {

// Shared layout: [0, 128) the table's barrier; table; thresholds; squared rp edges;
// scales of rp w; per warp a queue and a ring; per slot the count and
// [w lo, w hi, rp w lo, rp w hi], shared by the CTA's warps.
constexpr int SRP_QUEUE = (CRP_E2 + (NB_MAX + 1) * 8 + NB_MAX * 4 + 127) / 128 * 128;
constexpr int SRP_SR = CRP_E2 + (NB_MAX + 1) * 8;
constexpr int SRP_RING = SRP_QUEUE + WARPS * (int)sizeof(FlagQueue);
// Lane pairs of a warp between its flushes: 8 warps of 32 lanes adding terms of 2^41
// to one 64-bit sum stay below 2^63.
constexpr unsigned SRP_FLUSH = 1u << 13;

__device__ __forceinline__ void add_term(uint32_t *s, double *global, float v, float t)
{
    const uint32_t b = __float_as_uint(t);
    const unsigned sh = ((b >> 23) & 0xffu) - 150u;  // t = mantissa * 2^sh
    if (sh <= 18u) {
        u64 q = (u64)((b & 0x7fffffu) | 0x800000u) << sh;
        if ((int)b < 0)
            q = 0ull - q;
        const uint32_t lo = (uint32_t)q, old = atomicAdd(s, lo);
        const uint32_t hi = (uint32_t)(q >> 32) + (old + lo < old ? 1u : 0u);
        if (hi)
            atomicAdd(s + 1, hi);
    } else if (v != 0.0f) {
        atomicAdd(global, (double)v);
    }
}

// A counted pair's terms: pw its weight, sw the scale of w, rp2 the (corrected)
// squared separation.
template <bool W, bool RV>
__device__ __forceinline__ void add_slot(const PairParams &P, unsigned char *slots, const float *sr, int k, int m,
                                         float pw, float sw, float rp2)
{
    const int s = k * P.npibins + m;
    uint32_t *c = reinterpret_cast<uint32_t *>(slots) + 5 * s;
    atomicAdd(c, 1u);
    if (W)
        add_term(c + 1, P.wsum + s, pw, pw * sw);
    if (RV) {
        const float rw = W ? __fmul_rn(sqrt_approx(rp2), pw) : sqrt_approx(rp2);
        add_term(c + 3, P.rsum + s, rw, rw * sr[k]);
    }
}

template <bool W, bool RV, bool RL>
__device__ __noinline__ int settle_sums_rp(const PairParams &P, unsigned char *smem, unsigned char *slots,
                                           float sw, const FlagQueue *fq, int qn)
{
    const int lane = threadIdx.x & 31, first = max(0, qn - 32);
    int re = 0;
    __syncwarp();
    if (first + lane < qn) {
        const int i = fq->i[first + lane], j = fq->j[first + lane], im = fq->image[first + lane];
        const int qx = (im & 3) - 1, qy = ((im >> 2) & 3) - 1, qz = ((im >> 4) & 3) - 1;
        const RpPair r = rp_pair(P, smem, i, j, qx, qy, qz);
        const int s = rp_slot(P, smem, r, i, j, qx, qy, qz, re);
        if (s >= 0) {
            float rp2 = r.rp2;
            if (RL) {
                const float *a = P.A.xyz + quad_off((uint32_t)i), *b = P.B.xyz + quad_off((uint32_t)j);
                const float *ra = P.A.res + quad_off((uint32_t)i), *rb = P.B.res + quad_off((uint32_t)j);
                const float Sx = (float)qx * P.boxf[0], Sy = (float)qy * P.boxf[1];
                const float xh = __fsub_rn(a[0], Sx), yh = __fsub_rn(a[4], Sy);
                const float lx = shifted_residual(ra[0], a[0], Sx, xh, qx, P.boxr[0]);
                const float ly = shifted_residual(ra[4], a[4], Sy, yh, qy, P.boxr[1]);
                const float dx = __fsub_rn(b[0], xh), dy = __fsub_rn(b[4], yh);
                const float ex = __fsub_rn(rb[0], lx), ey = __fsub_rn(rb[4], ly);
                if (rp2 < P.near) {
                    const float cx = __fadd_rn(dx, ex), cy = __fadd_rn(dy, ey);
                    rp2 = __fmaf_rn(cy, cy, __fmul_rn(cx, cx));
                } else {
                    rp2 = __fmaf_rn(2.0f, __fmaf_rn(dy, ey, __fmul_rn(dx, ex)), rp2);
                }
            }
            const int k = s / (P.npibins + 1);
            add_slot<W, RV>(P, slots, reinterpret_cast<const float *>(smem + SRP_SR), k, s - k * (P.npibins + 1),
                            W ? __fmul_rn(P.B.ws[j], P.A.ws[i]) : 1.0f, sw, rp2);
        }
    }
    __syncwarp();
    return re;
}

// RL: rp^2 corrected to first order with the coordinates' float32 rounding residuals,
// rp2 = rp2~ + 2 (dx~ ex + dy~ ey), but of pairs with rp2~ < near from corrected
// differences (see sums32.cuh).
template <int PP, bool W, bool RV, bool RL, bool EVALS, bool LIN, bool SL = false>
struct SumsRp32 {
    static constexpr int I = 16, CH = I * PP, JS = 128 / I;
    using Ring = RingSums<W, RL>;
    static constexpr int SLOTS = SRP_RING + WARPS * Ring::BYTES;  // byte offset of the slots
    struct State {
        u64 n_eval, n_rck;
        unsigned pending;  // lane pairs since the warp's last flush
        int qn;            // flagged pairs waiting in the warp's queue
        float sw;          // scale of w
    };

    static __device__ __forceinline__ bool init(const PairParams &P, unsigned char *smem, State &st)
    {
        const int tid = threadIdx.x;
        if (tid == 0) {
            mbar_init(reinterpret_cast<uint64_t *>(smem), 1);
            fence_mbar_init();
        }
        __syncthreads();
        const float mw = W ? wmax_pair(P) : 1.0f;
        const bool ok = load_table(P, smem, CRP_LUT, 0u, [&]() {
            for (int q = tid; q < P.nthr; q += THREADS)
                reinterpret_cast<float *>(smem + CRP_THR)[q] = P.thr[q];
            for (int q = tid; q <= P.nbins; q += THREADS)
                reinterpret_cast<double *>(smem + CRP_E2)[q] = P.E2[q];
            for (int q = tid; q < P.nbins; q += THREADS)
                reinterpret_cast<float *>(smem + SRP_SR)[q] =
                    pow2_floor(1099511627776.0f / (sqrtf((float)P.E2[q + 1]) * mw));
            for (int q = tid; q < 5 * P.nbins * P.npibins; q += THREADS)
                reinterpret_cast<uint32_t *>(smem + SLOTS)[q] = 0u;
        });
        st = State{0ull, 0ull, 0u, 0, pow2_floor(1099511627776.0f / mw)};
        return ok;
    }

    // Slots s0, s0 + step, ... to the global results.  Other warps may be adding: each
    // word is taken by one exchange, so no term is lost (a carry on its way is
    // flushed by the next).
    static __device__ __noinline__ void flush(const PairParams &P, unsigned char *smem, float sw, int s0, int step)
    {
        uint32_t *acc = reinterpret_cast<uint32_t *>(smem + SLOTS);
        const float *sr = reinterpret_cast<const float *>(smem + SRP_SR);
        for (int s = s0; s < P.nbins * P.npibins; s += step) {
            const uint32_t c = atomicExch(acc + 5 * s, 0u);
            if (c)
                atomicAdd(&P.hist[s], (u64)c);
            for (int v = W ? 0 : 1; v < (RV ? 2 : 1); ++v) {
                uint32_t *w = acc + 5 * s + 1 + 2 * v;
                const uint32_t lo = atomicExch(w, 0u), hi = atomicExch(w + 1, 0u);
                const long long q = (long long)(((u64)hi << 32) | lo);
                if (q)
                    atomicAdd(v ? &P.rsum[s] : &P.wsum[s], (double)q / (double)(v ? sr[s / P.npibins] : sw));
            }
        }
    }

    template <bool TRI>
    static __device__ __forceinline__ void sweep(const PairParams &P, unsigned char *smem, State &st,
                                                 uint32_t addr, int j0, int j1, int jlo, int jhi, int jj, int ii,
                                                 const u64 (&XH)[PP], const u64 (&YH)[PP], const u64 (&ZH)[PP],
                                                 const u64 (&LX)[PP], const u64 (&LY)[PP], const u64 (&WI)[PP],
                                                 int ib, int image, unsigned vmask)
    {
        const u64 MG = pack2(PI_MAGIC, PI_MAGIC), LS = pack2(P.lut_scale, P.lut_scale),
                  LM = pack2(LIN_MAGIC, LIN_MAGIC), TWO = pack2(2.0f, 2.0f);
        const float sc = P.pscale, pband = P.pband;
        const uint32_t npi = (uint32_t)P.npibins, nbu = (uint32_t)P.nbins;
        const uint32_t lutb = smem_u32(smem + CRP_LUT), lut_lo = lutb - LIN_MAGIC_BITS,
                       lut_last = (uint32_t)(P.lut_n - 1), lut_hi = lutb + lut_last;
        const float *sr = reinterpret_cast<const float *>(smem + SRP_SR);
        const uint32_t p0 = addr + 48u * jj;  // this lane's first quad
        const int jf = j0 + 4 * jj;           // its first secondary
        FlagQueue *fq = reinterpret_cast<FlagQueue *>(smem + SRP_QUEUE) + (threadIdx.x >> 5);
        uint32_t p = p0, pw4 = addr + Ring::W_OFF + 16u * jj;
        for (int nit = (j1 - j0 + JS - 1) / JS; nit > 0; nit -= 8) {
            const int tend = min(8, nit);
            const uint32_t pb = p, pend = p + (uint32_t)tend * (12u * JS);
            uint32_t fm[PP];
#pragma unroll
            for (int q = 0; q < PP; ++q)
                fm[q] = 0u;
#pragma unroll 1
            for (; p != pend; p += 12 * JS, pw4 += 4 * JS) {
                const int jt = jf + (int)((p - p0) / 12u);  // (TRI and diagnostics only)
                ulonglong2 vx, vy, vz, rx, ry, wv;
                lds128<0>(p, vx);
                lds128<16>(p, vy);
                lds128<32>(p, vz);
                if (RL) {
                    lds128<Ring::RES_OFF>(p, rx);
                    lds128<Ring::RES_OFF + 16>(p, ry);
                }
                if (W)
                    lds128<0>(pw4, wv);
#pragma unroll
                for (int q = 0; q < PP; ++q) {
                    float r[4], rc[4], t[4], s[4], w[4], pw[4];
                    uint32_t cq[4];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const u64 dx = fsub2(h ? vx.y : vx.x, XH[q]), dy = fsub2(h ? vy.y : vy.x, YH[q]);
                        const u64 r2 = ffma2(dy, dy, fmul2(dx, dx));
                        float za, zb;
                        unpack2(fsub2(h ? vz.y : vz.x, ZH[q]), za, zb);
                        t[2 * h] = __fmaf_rn(fabsf(za), sc, -0.5f);
                        t[2 * h + 1] = __fmaf_rn(fabsf(zb), sc, -0.5f);
                        const u64 t2 = pack2(t[2 * h], t[2 * h + 1]);
                        const u64 s2 = fadd2(t2, MG);
                        unpack2(r2, r[2 * h], r[2 * h + 1]);
                        unpack2(s2, s[2 * h], s[2 * h + 1]);
                        unpack2(fsub2(t2, fsub2(s2, MG)), w[2 * h], w[2 * h + 1]);
                        if (RL)
                            unpack2(ffma2(TWO, ffma2(dy, fsub2(h ? ry.y : ry.x, LY[q]),
                                                     fmul2(dx, fsub2(h ? rx.y : rx.x, LX[q]))), r2),
                                    rc[2 * h], rc[2 * h + 1]);
                        if (W)
                            unpack2(fmul2(h ? wv.y : wv.x, WI[q]), pw[2 * h], pw[2 * h + 1]);
                        if (LIN) {
                            float c[2];
                            unpack2(ffma2(r2, LS, LM), c[0], c[1]);
                            cq[2 * h] = min(__float_as_uint(c[0]) + lut_lo, lut_hi);
                            cq[2 * h + 1] = min(__float_as_uint(c[1]) + lut_lo, lut_hi);
                        } else {
                            cq[2 * h] = lutb + min((__float_as_uint(r[2 * h]) >> P.lut_shift) - P.u0, lut_last);
                            cq[2 * h + 1] = lutb + min((__float_as_uint(r[2 * h + 1]) >> P.lut_shift) - P.u0,
                                                       lut_last);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        // sign set: near a pi edge (a NaN of the padding is positive)
                        float g = __fsub_rn(pband, fabsf(w[k]));
                        if (TRI) {  // pairs with j <= i: not counted, never flagged
                            const bool live = jt + k > ib + q * I + ii;
                            cq[k] = live ? cq[k] : lut_hi;
                            g = live ? g : 1.0f;
                        }
                        if (EVALS)
                            st.n_eval += (((vmask >> q) & 1u) && jt + k >= jlo && jt + k < jhi &&
                                          (!TRI || jt + k > ib + q * I + ii)) ? 1ull : 0ull;
                        const uint32_t e = lds_entry(cq[k]);
                        const uint32_t m = __float_as_uint(s[k]) - PI_MAGIC_BITS;
                        const uint32_t f = e | __float_as_uint(g);  // sign set: settled later
                        fm[q] = push_sign(fm[q], f);  // pair (t, k) ends at bit 4 tend - 1 - (4 t + k)
                        if ((int)f >= 0 && e < nbu && m < npi)
                            add_slot<W, RV>(P, smem + SLOTS, sr, (int)e, (int)m, W ? pw[k] : 1.0f, st.sw,
                                            RL ? rc[k] : r[k]);
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
                        if (st.qn >= 32)
                            settle(P, smem, st);
                    }
                }
            }
        }
    }

    static __device__ __forceinline__ void settle(const PairParams &P, unsigned char *smem, State &st)
    {
        st.n_rck += settle_sums_rp<W, RV, RL>(P, smem, smem + SLOTS, st.sw,
                                              reinterpret_cast<const FlagQueue *>(smem + SRP_QUEUE) +
                                                  (threadIdx.x >> 5), st.qn);
        st.qn = max(0, st.qn - 32);
        ++st.pending;
    }

    static __device__ __forceinline__ void task(const PairParams &P, unsigned char *smem, State &st,
                                                unsigned c, unsigned part, unsigned parts)
    {
        const int lane = threadIdx.x & 31, ii = lane % I, jj = lane / I;
        const uint32_t ring = smem_u32(smem + SRP_RING) + (threadIdx.x >> 5) * (uint32_t)Ring::BYTES;
        const int ib = (int)(c * CH);
        Chunk<I, PP> C;
        if (!C.load(P, ib, ii))
            return;
        u64 XH[PP], YH[PP], ZH[PP], LX[PP], LY[PP], WI[PP];
        float rx[PP], ry[PP];
#pragma unroll
        for (int q = 0; q < PP; ++q) {
            const int i = ib + q * I + ii;
            LX[q] = LY[q] = WI[q] = 0ull;
            rx[q] = ry[q] = 0.0f;
            if (W) {
                const float w = __ldg(P.A.ws + i);
                WI[q] = pack2(w, w);
            }
            if (RL) {
                const float *r = P.A.res + quad_off((uint32_t)i);
                rx[q] = __ldg(r);
                ry[q] = __ldg(r + 4);
            }
        }
        int image = 0;
        for_windows<JS, Ring, SL>(
            P, C.col, ib, C.zlo, C.zhi, (int)part, (int)parts, lane, ring,
            [&](int k, int code) {
                image = C.shift(P, k, code, XH, YH, ZH);
                if (RL) {
                    const int qx = (code & 3) - 1, qy = ((code >> 2) & 3) - 1;
                    const float Sx = (float)qx * P.boxf[0], Sy = (float)qy * P.boxf[1];
#pragma unroll
                    for (int q = 0; q < PP; ++q) {
                        float xh, yh, t;
                        unpack2(XH[q], xh, t);
                        unpack2(YH[q], yh, t);
                        const float lx = shifted_residual(rx[q], C.x[q], Sx, xh, qx, P.boxr[0]);
                        const float ly = shifted_residual(ry[q], C.y[q], Sy, yh, qy, P.boxr[1]);
                        LX[q] = pack2(lx, lx);
                        LY[q] = pack2(ly, ly);
                    }
                }
            },
            [&](uint32_t addr, int j0, int j1, int jlo, int jhi, bool tri) {
                st.pending += (unsigned)((j1 - j0) / JS + 1) * 4u * PP;
                if (tri)
                    sweep<true>(P, smem, st, addr, j0, j1, jlo, jhi, jj, ii, XH, YH, ZH, LX, LY, WI, ib, image,
                                C.vmask);
                else
                    sweep<false>(P, smem, st, addr, j0, j1, jlo, jhi, jj, ii, XH, YH, ZH, LX, LY, WI, ib, image,
                                 C.vmask);
                if (st.pending > SRP_FLUSH - Ring::N * PP) {
                    __syncwarp();
                    flush(P, smem, st.sw, lane, 32);
                    st.pending = 0u;
                }
            });
    }

    static __device__ __forceinline__ void fini(const PairParams &P, unsigned char *smem, State &st)
    {
        if (st.qn)
            settle(P, smem, st);
        __syncthreads();
        flush(P, smem, st.sw, (int)threadIdx.x, THREADS);
        const u64 n_rck = warp_sum_u64(st.n_rck), n_eval = EVALS ? warp_sum_u64(st.n_eval) : 0ull;
        if ((threadIdx.x & 31) == 0) {
            if (n_rck)
                atomicAdd(&P.diag[2], n_rck);
            if (n_eval)
                atomicAdd(&P.diag[1], n_eval);
        }
    }
};

}  // namespace

}  // namespace cf
