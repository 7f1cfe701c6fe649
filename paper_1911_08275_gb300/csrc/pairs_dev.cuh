// Device code shared by the pair kernels: packed float32 arithmetic, searches,
// binary64 evaluation, table and histogram helpers, column-pair planning.
#pragma once

#include <cuda_runtime.h>

#include "cf_internal.cuh"

namespace cf {

namespace {

typedef unsigned long long u64;

__device__ __forceinline__ int floor_div(int a, int n)
{
    return a >= 0 ? a / n : -((-a + n - 1) / n);
}

// ---------------------------------------------------------------- packed f32x2
__device__ __forceinline__ u64 pack2(float lo, float hi)
{
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(u64 v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ u64 fsub2(u64 a, u64 b)
{
    u64 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ u64 fadd2(u64 a, u64 b)
{
    u64 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ u64 fmul2(u64 a, u64 b)
{
    u64 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ u64 ffma2(u64 a, u64 b, u64 c)
{
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// ---------------------------------------------------------------- searches
// Bin of a binary64 squared separation: k with E2[k] <= r2 < E2[k+1], else -1.
// Non-negative doubles order like their bit patterns, so integer compares suffice.
__device__ __forceinline__ int bin_f64(double r2, const double *E2, int nb)
{
    const long long u = __double_as_longlong(r2);
    const long long *e = reinterpret_cast<const long long *>(E2);
    if (!(u >= e[0] && u < e[nb]))
        return -1;
    int lo = 0, hi = nb;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (e[mid] <= u)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

__device__ __forceinline__ double canon_r2(const double4_32a &p, const double4_32a &q, double Sx,
                                           double Sy, double Sz)
{
    const double dx = canon_comp(p.x, q.x, Sx);
    const double dy = canon_comp(p.y, q.y, Sy);
    const double dz = canon_comp(p.z, q.z, Sz);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// Debug: does the float32 decision for d2 agree with binary64?  (1 = violation)
__device__ __noinline__ int verify_pair(float d2, const float *thr, int nthr, int nb,
                                        const double *E2, const double4_32a *pa,
                                        const double4_32a *pb, int i, int j, double Sx, double Sy,
                                        double Sz)
{
    int c = 0;
    while (c < nthr && thr[c] <= d2)
        ++c;
    if (c & 1)
        return 0;  // inside a band: re-checked, no float32 claim
    const int k32 = (c >= 2 && c <= 2 * nb) ? (c - 2) >> 1 : -1;
    const int k64 = bin_f64(canon_r2(pa[i], pb[j], Sx, Sy, Sz), E2, nb);
    return k32 != k64;
}

__device__ __forceinline__ u64 warp_sum_u64(u64 v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(FULL, v, o);
    return v;
}

// Move a copy's counts (a word per lane and bin) to the global histogram while other warps
// add to it: each count is read and cleared in one atomic exchange, so no increment is lost.
__device__ void warp_flush_shared(uint32_t *hw, int nb, unsigned long long *ghist, int lane)
{
    for (int b = 0; b < nb; ++b) {
        const u64 v = warp_sum_u64(atomicExch(&hw[b * 32 + lane], 0u));
        if (lane == 0 && v)
            atomicAdd(&ghist[b], v);
    }
}

// Cells linear in d2: adding 2^23 in the fma rounds d2 * scale to an integer q
// held in the sum's low bits (exact below 2^22; larger values, and NaN, give
// larger bit patterns and clamp to the out-of-range entry).
constexpr float LIN_MAGIC = 8388608.0f;  // 2^23: spacing 1 in [2^23, 2^24)
constexpr uint32_t LIN_MAGIC_BITS = 0x4b000000u;

// Number of thresholds T[c] <= d2 (T is non-decreasing; NaN counts none).
__device__ __forceinline__ int thr_count(const float *T, int nthr, float d2)
{
    int lo = 0, hi = nthr;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (T[mid] <= d2)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}

__device__ __forceinline__ void red_shared1(uint32_t addr)
{
    asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(addr));
}

// Table byte at a shared address, sign-extended: the flagged entry gives -1.
__device__ __forceinline__ uint32_t lds_entry(uint32_t addr)
{
    uint32_t e;
    asm volatile("ld.shared.s8 %0, [%1];" : "=r"(e) : "r"(addr));
    return e;
}

// 16-byte shared load (four floats as two packed pairs) at a 32-bit shared
// address plus a constant offset.
template <int OFF>
__device__ __forceinline__ void lds128(uint32_t a, ulonglong2 &v)
{
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2+%3];" : "=l"(v.x), "=l"(v.y) : "r"(a), "n"(OFF));
}

// (m << 1) | (v >> 31): one funnel shift appends v's sign bit to the mask m.
__device__ __forceinline__ uint32_t push_sign(uint32_t m, uint32_t v)
{
    uint32_t r;
    asm("shf.l.wrap.b32 %0, %1, %2, 1;" : "=r"(r) : "r"(v), "r"(m));
    return r;
}

// Candidate (column a, stencil offset) -> column pair, image, pruning
// (Sec. 2.2) in binary64 and z reach.  Returns false if the pair has no work.
__device__ __forceinline__ bool plan_item(const PairParams &P, int item, Nbr &w)
{
    const int a = item / P.nstencil, s = item - a * P.nstencil;
    const int2 o = P.stencil[s];
    const int ax = a / P.g.ncy, ay = a - ax * P.g.ncy;
    int bx = ax + o.x, by = ay + o.y;
    int qx = 0, qy = 0;
    if (P.g.periodic) {
        qx = floor_div(bx, P.g.ncx);
        qy = floor_div(by, P.g.ncy);
        // an image two or more boxes away holds no pair within Rmax < L/2 (every
        // coordinate difference is below L), even when pruning is switched off
        if (qx < -1 || qx > 1 || qy < -1 || qy > 1)
            return false;
        bx -= qx * P.g.ncx;
        by -= qy * P.g.ncy;
    } else if (bx < 0 || bx >= P.g.ncx || by < 0 || by >= P.g.ncy) {
        return false;
    }
    const int b = bx * P.g.ncy + by;
    const long long nz = P.g.nz;
    if (P.shard_n > 1) {  // deterministic split of the primary columns over shards
        const unsigned long long total = P.A.cell_start[(long long)P.g.ncols * nz];
        const unsigned long long first = P.A.cell_start[a * nz];
        const unsigned long long lo = total * (unsigned long long)P.shard_k / P.shard_n;
        const unsigned long long hi = total * (unsigned long long)(P.shard_k + 1) / P.shard_n;
        if (first < lo || first >= hi)
            return false;
    }
    if (P.A.cell_start[a * nz] >= P.A.cell_start[(a + 1) * nz] || P.B.cell_start[b * nz] >= P.B.cell_start[(b + 1) * nz])
        return false;
    // minimum possible (x, y) separation of the two columns' bounding boxes; signs and
    // compares on the bits (the binary64 pipe is narrow)
    const ColBox ba = P.A.colbox[a], bb = P.B.colbox[b];
    auto gap = [](double a0, double a1, double b0, double b1, int q, double box) {
        if (q) {
            const double S = q > 0 ? box : -box;
            b0 = __dadd_rn(b0, S);
            b1 = __dadd_rn(b1, S);
        }
        const double up = __dsub_rn(b0, a1), dn = __dsub_rn(a0, b1);
        return __double_as_longlong(up) > 0 ? up : __double_as_longlong(dn) > 0 ? dn : 0.0;
    };
    const double gx = gap(key_value(ba.x0), key_value(ba.x1), key_value(bb.x0), key_value(bb.x1), qx, P.g.box[0]);
    const double gy = gap(key_value(ba.y0), key_value(ba.y1), key_value(bb.y0), key_value(bb.y1), qy, P.g.box[1]);
    const double g2 = __dadd_rn(__dmul_rn(gx, gx), __dmul_rn(gy, gy));
    if (!(P.flags & CF_FLAG_NO_PRUNE) && __double_as_longlong(g2) >= __double_as_longlong(P.prune_r2))
        return false;
    // z reach, rounded up: dz_max,all of Sec. 2.2 (xi); pimax (rp-pi)
    if (P.kind == 0) {
        const double t = __dsub_rn(P.rxy2, __dmul_rn(g2, 1.0 - 1e-12));
        w.dz = __double_as_longlong(t) > 0 ? __fmul_ru(__fsqrt_ru(__double2float_ru(t)), 1.0f + 0x1p-22f) : 0.0f;
    } else {
        w.dz = __double2float_ru(P.rz);
    }
    w.dz = __fadd_ru(w.dz, P.zslack);
    const bool self = P.autocorr && o.x == 0 && o.y == 0;
    w.code = (qx + 1) | ((qy + 1) << 2) | (self ? 16 : 0) | (b << 5);
    return true;
}

}  // namespace

}  // namespace cf
