// Float32 DD(r) with pair weights and / or mean separations over chunk tasks
// (tasks.cuh): the sweep of count32.cuh with two more shared rows per bin.
//
// A pair adds round(v * scale) for its weight v = w_i w_j (scale sw) and for r v (a
// scale per bin) to 32-bit words of its lane, as the low mantissa bits of
// fma(v, scale, 1.5 * 2^23): a word then holds count * bits(1.5 * 2^23) plus the exact
// integer sum, which the lane's own count recovers.  Scales are powers of two
// with every term at most 2^21 in size, so 1023 terms cannot overflow; before that a
// warp moves its words to 64-bit sums of the CTA, one bin per lane.  The rounding
// error of one term is at most half a unit: relative to the term 2^-22
// max|w_i w_j| / |w_i w_j| (times e_{k+1} / e_k for r w).
//
// The words of a bin and lane lie 128 bytes apart (count, w, r w), so one address
// serves the three atomics; weights and coordinate residuals come through the
// warp's ring with the coordinates, not from global memory in the loop.
//
// Bound, and what was measured:
// 1.2M x 12M points, open box, 20 bins (4.2e10 evaluations, GB300): weights and mean r
// 67.6 -> 44.8 ms, weights alone 37.0 -> 25.9 ms, 211 instructions per step of 8
// pairs per lane (266 before), issue 62 % (44), the L1's data path 74 % busy: both
// bind.  300k points, weights: 0.40 -> 0.22 ms (the 64-bit sums were 37 MB of
// per-thread scratch, cleared and merged in every call).
#pragma once

#include <type_traits>

#include "tasks.cuh"

namespace cf {

namespace {

constexpr float QMAGIC = 12582912.0f;  // 1.5 * 2^23
constexpr uint32_t QMAGIC_BITS = 0x4b400000u;
constexpr unsigned SUM_TERMS = 1023;   // terms a word may hold

// Shared layout: [0, 128) the table's barrier; table; thresholds; squared edges;
// scales of r w (rows -1 .. nbins); 64-bit sums [bin][count, w, r w] of the CTA; per
// warp a queue of flagged pairs and a ring; words [warp][row][plane][lane].
constexpr int S32_LUT = 128;
constexpr int S32_THR = S32_LUT + LUT_MAX;
constexpr int S32_E2 = S32_THR + 2 * (NB_MAX + 1) * 4;
constexpr int S32_SR = S32_E2 + (NB_MAX + 1) * 8;
constexpr int S32_QUEUE = (S32_SR + (NB_MAX + 2) * 4 + 127) / 128 * 128;
constexpr int S32_ACC = S32_QUEUE + WARPS * (int)sizeof(FlagQueue);

template <bool W, bool RV, bool RL>
struct SumLayout {
    static constexpr int PLANES = 1 + (W ? 1 : 0) + (RV ? 1 : 0);
    static constexpr int ROW = PLANES * 128;  // bytes
    using Ring = RingSums<W, RL>;
    static __host__ __device__ int ring(int nb) { return align_up(S32_ACC + nb * 24, 128); }
    static __host__ __device__ int words(int nb) { return ring(nb) + WARPS * Ring::BYTES; }
    static __host__ __device__ int total(int nb) { return words(nb) + WARPS * (nb + 2) * ROW; }
};

template <int OFF>
__device__ __forceinline__ void red_shared_at(uint32_t addr, uint32_t v)
{
    asm volatile("red.shared.add.u32 [%0+%2], %1;" ::"r"(addr), "r"(v), "n"(OFF));
}

__device__ __forceinline__ float lds_f32(uint32_t addr)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}

__device__ __forceinline__ float pow2_floor(float x)
{
    return (x > 0.0f && x < INFINITY) ? __uint_as_float(__float_as_uint(x) & 0x7f800000u) : 1.0f;
}

__device__ __forceinline__ float wmax_pair(const PairParams &P)
{
    return __uint_as_float(*P.A.wmax) * __uint_as_float(*P.B.wmax);
}

// Rounding error of s = fl(a + b), i.e. a + b - s exactly (Knuth's TwoSum).
__device__ __forceinline__ float two_sum_err(float a, float b, float s)
{
    const float bb = __fsub_rn(s, a);
    return __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

__device__ __forceinline__ float sqrt_approx(float v)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// A primary's residual along one axis after the shift by q boxes:
// r + (x - S - x^) - (q L - fl32(q L)), x^ = fl32(x - S).
__device__ __forceinline__ float shifted_residual(float r, float x, float S, float xh, int q, float boxr)
{
    return __fsub_rn(__fadd_rn(r, two_sum_err(x, -S, xh)), (float)q * boxr);
}

// What the adds need.
struct SumState {
    uint32_t hl;     // shared address of this lane's count word of row 0
    uint32_t srb;    // shared address of the r w scale of row 0
    float sw;        // scale of w
    FlagQueue *fq;
    int qn;          // flagged pairs waiting in the warp's queue
    unsigned wpend;  // terms a word may hold since the last flush, at most
    u64 n_eval, n_rck;
};

template <bool W, bool RV>
__device__ __forceinline__ void sum_add(uint32_t hl, uint32_t srb, float sw, uint32_t e, float pw, float d2)
{
    const uint32_t a = hl + e * (uint32_t)SumLayout<W, RV, false>::ROW;
    red_shared1(a);
    if (W)
        red_shared_at<128>(a, __float_as_uint(__fmaf_rn(pw, sw, QMAGIC)));
    if (RV) {
        const float r = sqrt_approx(d2);
        const float rw = W ? __fmul_rn(r, pw) : r;
        red_shared_at<W ? 256 : 128>(a, __float_as_uint(__fmaf_rn(rw, lds_f32(srb + e * 4u), QMAGIC)));
    }
}

// Move the warp's words of the counted bins to the CTA's 64-bit sums: lane b takes
// bin b, reading the lanes' words in an order that gives every lane its own bank.
template <bool W, bool RV>
__device__ __noinline__ void sum_flush(unsigned char *words, unsigned long long *acc, int nb)
{
    constexpr int PLANES = SumLayout<W, RV, false>::PLANES;
    const int lane = threadIdx.x & 31;
    uint32_t *h = reinterpret_cast<uint32_t *>(words);
    __syncwarp();
    for (int b = lane; b < nb; b += 32) {
        long long c = 0, w = 0, r = 0;
        for (int l = 0; l < 32; ++l) {
            uint32_t *p = h + (b + 1) * PLANES * 32 + ((l + lane) & 31);
            const uint32_t n = p[0];
            p[0] = 0u;
            c += n;
            if (W) {
                w += (int)(p[32] - n * QMAGIC_BITS);
                p[32] = 0u;
            }
            if (RV) {
                r += (int)(p[W ? 64 : 32] - n * QMAGIC_BITS);
                p[W ? 64 : 32] = 0u;
            }
        }
        if (c) {
            atomicAdd(acc + 3 * b, (u64)c);
            if (W)
                atomicAdd(acc + 3 * b + 1, (u64)w);
            if (RV)
                atomicAdd(acc + 3 * b + 2, (u64)r);
        }
    }
    __syncwarp();
}

// Settle the last min(32, qn) flagged pairs of the warp's queue, one per lane (as
// count32.cuh's settle), with their sums.
template <bool W, bool RV, bool RL>
__device__ __noinline__ int settle_sums(const PairParams &P, const unsigned char *smem, uint32_t hl,
                                        uint32_t srb, float sw, const FlagQueue *fq, int qn)
{
    const int lane = threadIdx.x & 31, first = max(0, qn - 32);
    int row = -1, re = 0;
    float pw = 1.0f, dc = 0.0f;
    __syncwarp();
    if (first + lane < qn) {
        const int i = fq->i[first + lane], j = fq->j[first + lane], m = fq->image[first + lane];
        const int qx = (m & 3) - 1, qy = ((m >> 2) & 3) - 1, qz = ((m >> 4) & 3) - 1;
        const float *a = P.A.xyz + quad_off((uint32_t)i), *b = P.B.xyz + quad_off((uint32_t)j);
        const float Sx = (float)qx * P.boxf[0], Sy = (float)qy * P.boxf[1], Sz = (float)qz * P.boxf[2];
        const float xh = __fsub_rn(a[0], Sx), yh = __fsub_rn(a[4], Sy), zh = __fsub_rn(a[8], Sz);
        const float dx = __fsub_rn(b[0], xh), dy = __fsub_rn(b[4], yh), dz = __fsub_rn(b[8], zh);
        const float d2 = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
        dc = d2;
        if (RL) {
            const float *ra = P.A.res + quad_off((uint32_t)i), *rb = P.B.res + quad_off((uint32_t)j);
            const float lx = shifted_residual(ra[0], a[0], Sx, xh, qx, P.boxr[0]);
            const float ly = shifted_residual(ra[4], a[4], Sy, yh, qy, P.boxr[1]);
            const float lz = shifted_residual(ra[8], a[8], Sz, zh, qz, P.boxr[2]);
            const float ex = __fsub_rn(rb[0], lx), ey = __fsub_rn(rb[4], ly), ez = __fsub_rn(rb[8], lz);
            dc = __fmaf_rn(2.0f, __fmaf_rn(dz, ez, __fmaf_rn(dy, ey, __fmul_rn(dx, ex))), d2);
            if (d2 < P.near) {
                const float cx = __fadd_rn(dx, ex), cy = __fadd_rn(dy, ey), cz = __fadd_rn(dz, ez);
                dc = __fmaf_rn(cz, cz, __fmaf_rn(cy, cy, __fmul_rn(cx, cx)));
            }
        }
        if (W)
            pw = __fmul_rn(P.B.ws[j], P.A.ws[i]);
        const int c = thr_count(reinterpret_cast<const float *>(smem + S32_THR), P.nthr, d2);
        if (!(c & 1)) {
            row = (c >= 2 && c <= 2 * P.nbins) ? (c - 2) >> 1 : -1;
        } else {
            row = bin_f64(canon_r2(P.A.pos64[i], P.B.pos64[j], (double)qx * P.g.box[0],
                                   (double)qy * P.g.box[1], (double)qz * P.g.box[2]),
                          reinterpret_cast<const double *>(smem + S32_E2), P.nbins);
            re = 1;
        }
    }
    if (row >= 0)
        sum_add<W, RV>(hl, srb, sw, (uint32_t)row, pw, dc);
    __syncwarp();
    return re;
}

// RL: r from the squared distance corrected with the coordinates' float32 rounding
// residuals, d2 = d2~ + 2 (dx~ ex + dy~ ey + dz~ ez) up to the square of the residuals
// (primaries' residuals include the roundings of the shift).  Of points no farther apart
// than their residuals that square is all there is, and the sum negative: pairs with
// d2~ < near are flagged in the table, and the settling adds up corrected differences.
template <int PP, bool W, bool RV, bool RL, bool EVALS, int LT, bool SL = false>
struct Sums32 {
    static constexpr int I = 16, CH = I * PP, JS = 128 / I;
    using Lay = SumLayout<W, RV, RL>;
    using Ring = typename Lay::Ring;
    using State = SumState;

    static __device__ __forceinline__ unsigned char *words(const PairParams &P, unsigned char *smem)
    {
        return smem + Lay::words(P.nbins) + (threadIdx.x >> 5) * (P.nbins + 2) * Lay::ROW;
    }

    static __device__ __forceinline__ bool init(const PairParams &P, unsigned char *smem, State &st)
    {
        const int nb = P.nbins, tid = threadIdx.x;
        if (tid == 0) {
            mbar_init(reinterpret_cast<uint64_t *>(smem), 1);
            fence_mbar_init();
        }
        __syncthreads();
        const float mw = W ? wmax_pair(P) : 1.0f;
        const bool ok = load_table(P, smem, S32_LUT, 0u, [&]() {
            for (int q = tid; q < P.nthr; q += THREADS)
                reinterpret_cast<float *>(smem + S32_THR)[q] = P.thr[q];
            for (int q = tid; q <= nb; q += THREADS)
                reinterpret_cast<double *>(smem + S32_E2)[q] = P.E2[q];
            for (int k = tid; k < nb + 2; k += THREADS)  // r w < 2^20 scale in bin k - 1 (headroom 2)
                reinterpret_cast<float *>(smem + S32_SR)[k] =
                    (k >= 1 && k <= nb) ? pow2_floor(1048576.0f / (sqrtf((float)P.E2[k]) * mw)) : 0.0f;
            for (int q = tid; q < 3 * nb; q += THREADS)
                reinterpret_cast<unsigned long long *>(smem + S32_ACC)[q] = 0ull;
            uint32_t *h = reinterpret_cast<uint32_t *>(smem + Lay::words(nb));
            for (int q = tid; q < WARPS * (nb + 2) * Lay::ROW / 4; q += THREADS)
                h[q] = 0u;
        });
        st.hl = smem_u32(words(P, smem)) + Lay::ROW + (tid & 31) * 4;  // row 0 (row -1 before it)
        st.srb = smem_u32(smem + S32_SR) + 4;
        st.sw = W ? pow2_floor(2097152.0f / mw) : 1.0f;
        st.fq = reinterpret_cast<FlagQueue *>(smem + S32_QUEUE) + (tid >> 5);
        st.qn = 0;
        st.wpend = 0u;
        st.n_eval = st.n_rck = 0ull;
        return ok;
    }

    static __device__ __forceinline__ void flush(const PairParams &P, unsigned char *smem, State &st)
    {
        sum_flush<W, RV>(words(P, smem), reinterpret_cast<unsigned long long *>(smem + S32_ACC), P.nbins);
        st.wpend = 0u;
    }

    static __device__ __forceinline__ void settle(const PairParams &P, unsigned char *smem, State &st)
    {
        if (++st.wpend > SUM_TERMS) {  // a settled pair is one more term of a word
            flush(P, smem, st);
            st.wpend = 1u;
        }
        st.n_rck += settle_sums<W, RV, RL>(P, smem, st.hl, st.srb, st.sw, st.fq, st.qn);
        st.qn = max(0, st.qn - 32);
    }

    template <bool TRI, bool LIN>
    static __device__ __forceinline__ void sweep(const PairParams &P, unsigned char *smem, State &st,
                                                 uint32_t addr, int j0, int j1, int jlo, int jhi, int jj, int ii,
                                                 const u64 (&XH)[PP], const u64 (&YH)[PP], const u64 (&ZH)[PP],
                                                 const u64 (&LX)[PP], const u64 (&LY)[PP], const u64 (&LZ)[PP],
                                                 const u64 (&WI)[PP], int ib, int image, unsigned vmask)
    {
        const u64 LS = pack2(P.lut_scale, P.lut_scale), LM = pack2(LIN_MAGIC, LIN_MAGIC);
        const u64 TWO = pack2(2.0f, 2.0f);
        const uint32_t lutb = smem_u32(smem + S32_LUT), lut_lo = lutb - LIN_MAGIC_BITS,
                       lut_last = (uint32_t)(P.lut_n - 1), lut_hi = lutb + lut_last;
        const uint32_t p0 = addr + 48u * jj;  // this lane's first quad
        const int jf = j0 + 4 * jj;           // its first secondary
        uint32_t p = p0, pw4 = addr + Ring::W_OFF + 16u * jj;
        for (int nit = (j1 - j0 + JS - 1) / JS; nit > 0; nit -= 8) {
            const int tend = min(8, nit);
            const uint32_t pb = p, pend = p + (uint32_t)tend * (12u * JS);
            st.wpend += (unsigned)tend * 4u * PP;
            if (st.wpend > SUM_TERMS) {
                flush(P, smem, st);
                st.wpend = (unsigned)tend * 4u * PP;
            }
            uint32_t fm[PP];
#pragma unroll
            for (int q = 0; q < PP; ++q)
                fm[q] = 0u;
#pragma unroll 1
            for (; p != pend; p += 12 * JS, pw4 += 4 * JS) {
                const int jt = jf + (int)((p - p0) / 12u);  // (TRI and diagnostics only)
                ulonglong2 vx, vy, vz, rx, ry, rz, wv;
                lds128<0>(p, vx);
                lds128<16>(p, vy);
                lds128<32>(p, vz);
                if (RL) {
                    lds128<Ring::RES_OFF>(p, rx);
                    lds128<Ring::RES_OFF + 16>(p, ry);
                    lds128<Ring::RES_OFF + 32>(p, rz);
                }
                if (W)
                    lds128<0>(pw4, wv);
#pragma unroll
                for (int q = 0; q < PP; ++q) {
                    float d[4], dr[4], pw[4];
                    uint32_t cq[4];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const u64 dx = fsub2(h ? vx.y : vx.x, XH[q]), dy = fsub2(h ? vy.y : vy.x, YH[q]),
                                  dz = fsub2(h ? vz.y : vz.x, ZH[q]);
                        const u64 d2 = ffma2(dz, dz, ffma2(dy, dy, fmul2(dx, dx)));
                        unpack2(d2, d[2 * h], d[2 * h + 1]);
                        if (RL) {
                            const u64 c = ffma2(dz, fsub2(h ? rz.y : rz.x, LZ[q]),
                                                ffma2(dy, fsub2(h ? ry.y : ry.x, LY[q]),
                                                      fmul2(dx, fsub2(h ? rx.y : rx.x, LX[q]))));
                            unpack2(ffma2(TWO, c, d2), dr[2 * h], dr[2 * h + 1]);
                        }
                        if (W)
                            unpack2(fmul2(h ? wv.y : wv.x, WI[q]), pw[2 * h], pw[2 * h + 1]);
                        if (LIN) {
                            float c[2];
                            unpack2(ffma2(d2, LS, LM), c[0], c[1]);
                            cq[2 * h] = min(__float_as_uint(c[0]) + lut_lo, lut_hi);
                            cq[2 * h + 1] = min(__float_as_uint(c[1]) + lut_lo, lut_hi);
                        } else {
                            cq[2 * h] = lutb + min((__float_as_uint(d[2 * h]) >> P.lut_shift) - P.u0, lut_last);
                            cq[2 * h + 1] = lutb + min((__float_as_uint(d[2 * h + 1]) >> P.lut_shift) - P.u0,
                                                       lut_last);
                        }
                    }
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        if (TRI)
                            cq[r] = jt + r > ib + q * I + ii ? cq[r] : lut_hi;
                        if (EVALS)
                            st.n_eval += (((vmask >> q) & 1u) && jt + r >= jlo && jt + r < jhi &&
                                          (!TRI || jt + r > ib + q * I + ii)) ? 1ull : 0ull;
                        const uint32_t e = lds_entry(cq[r]);  // the row: bin, dummy or flagged (-1)
                        sum_add<W, RV>(st.hl, st.srb, st.sw, e, W ? pw[r] : 1.0f, RL ? dr[r] : d[r]);
                        fm[q] = push_sign(fm[q], e);  // pair (t, r) ends at bit 4 tend - 1 - (4 t + r)
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
                            const int b = 4 * tend - __ffs(m);  // = 4 t + r
                            const int at = st.qn + __popc(bm & ((1u << (threadIdx.x & 31)) - 1u));
                            st.fq->i[at] = ib + q * I + ii;
                            st.fq->j[at] = jf + (int)((pb - p0) / 12u) + (b >> 2) * JS + (b & 3);
                            st.fq->image[at] = image;
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

    static __device__ __forceinline__ void task(const PairParams &P, unsigned char *smem, State &st,
                                                unsigned c, unsigned part, unsigned parts)
    {
        const int lane = threadIdx.x & 31, ii = lane % I, jj = lane / I;
        const uint32_t ring = smem_u32(smem + Lay::ring(P.nbins)) + (threadIdx.x >> 5) * (uint32_t)Ring::BYTES;
        const int ib = (int)(c * CH);
        Chunk<I, PP> C;
        if (!C.load(P, ib, ii))
            return;
        u64 XH[PP], YH[PP], ZH[PP], LX[PP], LY[PP], LZ[PP], WI[PP];
        float rx[PP], ry[PP], rz[PP];
#pragma unroll
        for (int q = 0; q < PP; ++q) {
            const int i = ib + q * I + ii;
            LX[q] = LY[q] = LZ[q] = WI[q] = 0ull;
            rx[q] = ry[q] = rz[q] = 0.0f;
            if (W) {
                const float w = __ldg(P.A.ws + i);
                WI[q] = pack2(w, w);
            }
            if (RL) {
                const float *r = P.A.res + quad_off((uint32_t)i);
                rx[q] = __ldg(r);
                ry[q] = __ldg(r + 4);
                rz[q] = __ldg(r + 8);
            }
        }
        int image = 0;
        for_windows<JS, Ring, SL>(
            P, C.col, ib, C.zlo, C.zhi, (int)part, (int)parts, lane, ring,
            [&](int k, int code) {
                image = C.shift(P, k, code, XH, YH, ZH);
                if (RL) {
                    const int qx = (code & 3) - 1, qy = ((code >> 2) & 3) - 1;
                    const float Sx = (float)qx * P.boxf[0], Sy = (float)qy * P.boxf[1], Sz = (float)k * P.boxf[2];
#pragma unroll
                    for (int q = 0; q < PP; ++q) {
                        float xh, yh, zh, t;
                        unpack2(XH[q], xh, t);
                        unpack2(YH[q], yh, t);
                        unpack2(ZH[q], zh, t);
                        const float lx = shifted_residual(rx[q], C.x[q], Sx, xh, qx, P.boxr[0]);
                        const float ly = shifted_residual(ry[q], C.y[q], Sy, yh, qy, P.boxr[1]);
                        const float lz = shifted_residual(rz[q], C.z[q], Sz, zh, k, P.boxr[2]);
                        LX[q] = pack2(lx, lx);
                        LY[q] = pack2(ly, ly);
                        LZ[q] = pack2(lz, lz);
                    }
                }
            },
            [&](uint32_t addr, int j0, int j1, int jlo, int jhi, bool tri) {
                auto go = [&](auto tr, auto li) {
                    sweep<decltype(tr)::value, decltype(li)::value>(P, smem, st, addr, j0, j1, jlo, jhi, jj, ii,
                                                                    XH, YH, ZH, LX, LY, LZ, WI, ib, image, C.vmask);
                };
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
            });
    }

    static __device__ __forceinline__ void fini(const PairParams &P, unsigned char *smem, State &st)
    {
        if (st.qn)
            settle(P, smem, st);
        flush(P, smem, st);
        __syncthreads();
        const float *sr = reinterpret_cast<const float *>(smem + S32_SR) + 1;
        const long long *acc = reinterpret_cast<const long long *>(smem + S32_ACC);
        for (int b = threadIdx.x; b < P.nbins; b += THREADS)
            if (acc[3 * b]) {
                atomicAdd(&P.hist[b], (u64)acc[3 * b]);
                if (W)
                    atomicAdd(&P.wsum[b], (double)acc[3 * b + 1] / (double)st.sw);
                if (RV)
                    atomicAdd(&P.rsum[b], (double)acc[3 * b + 2] / (double)sr[b]);
            }
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
