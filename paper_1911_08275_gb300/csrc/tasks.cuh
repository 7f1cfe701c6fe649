// Chunk tasks: how the pair kernels walk the pairs of columns.
//
// A task is a run of CH z-consecutive points of one column of d1 (a chunk, held
// in the registers of one warp) against one share of that column's neighbour
// list (the kept column pairs of k_neighbours).  For each neighbour and
// periodic z image the warp finds the window of points whose z can lie within
// the pair's reach of the chunk (late entry / early exit of Sec. 2.2, Code 2,
// per chunk; one neighbour per lane), then sweeps the windows one after the
// other, the secondaries copied piece by piece into the warp's own part of shared
// memory one piece ahead.  Nothing is shared between the warps
// but the tables and the histogram, so there is no barrier between tasks and a
// column may be as narrow as a chunk.
#pragma once

#include <algorithm>
#include <type_traits>

#include "launch.cuh"
#include "pairs.cuh"
#include "pairs_dev.cuh"

namespace cf {

namespace {
// z of entry p in the quad layout.
__device__ __forceinline__ float quad_z(const float *__restrict__ q, int p)
{
    return __ldg(q + quad_off((uint32_t)p) + 8);
}

// Flagged pairs waiting to be settled (one queue per warp; at most 31 wait when
// up to 32 more are pushed).
struct FlagQueue {
    int i[64], j[64], image[64];
};

// Tasks of nchunk chunks: one task per chunk, but the last eighth of the chunks
// (TASK_TAIL) is split into parts, so that the last tasks to finish are short while
// most chunks pay the set-up of a task once.  All chunks are split where there
// are few (at most two per warp of the grid).  Measured on 1.2M points (kernel, ms at
// Rmax 5 / 10 / 25 / 50): every chunk in one part 0.218 / 0.288 / 1.248 / 5.600,
// every chunk in two 0.246 / 0.305 / 1.231 / 5.462; then, with the queue of flagged
// pairs, a tail of a quarter in 4 parts 0.232 / 0.280 / 1.135 / 5.166, of an eighth
// in 4 parts 0.219 / 0.271 / 1.127 / 5.162, in 8 parts 0.222 / 0.269 / 1.130 / 5.139.
constexpr unsigned TASK_TAIL = 8;
struct TaskSplit {
    unsigned whole, parts, ntask;
    __device__ TaskSplit(unsigned nchunk, unsigned parts_, bool all)
        : whole(parts_ == 1u ? nchunk : all ? 0u : nchunk - nchunk / TASK_TAIL), parts(parts_),
          ntask(whole + (nchunk - whole) * parts_)
    {
    }
    __device__ __forceinline__ void task(unsigned t, unsigned &chunk, unsigned &part, unsigned &nparts) const
    {
        chunk = t;
        part = 0;
        nparts = 1;
        if (t >= whole) {
            const unsigned s = (t - whole) / parts;
            chunk = whole + s;
            part = t - whole - s * parts;
            nparts = parts;
        }
    }
};

// The window of a column's entries with wlo <= z <= whi: [lo, hi) with lo the first
// entry with !(z < wlo) and hi the first with !(z <= whi).  The column is sorted by
// z (NaN padding at its end compares as larger than every value) and split into
// nz z-cells (offsets cs[0 .. nz]) by the gridding's monotone rule cell_index_f,
// so each bound lies in its value's cell and only that cell is searched; the two
// searches advance together, their loads in flight at the same time.
__device__ __forceinline__ void zwindow(const float *__restrict__ q, const uint32_t *__restrict__ cs, int nz,
                                        float inv_wz, float wlo, float whi, int &lo, int &hi)
{
    const int ca = cell_index_f(wlo, inv_wz, nz), cb = cell_index_f(whi, inv_wz, nz);
    int a0 = (int)__ldg(cs + ca), a1 = (int)__ldg(cs + ca + 1);
    int b0 = (int)__ldg(cs + cb), b1 = (int)__ldg(cs + cb + 1);
    while (a0 < a1 || b0 < b1) {
        const int ma = (a0 + a1) >> 1, mb = (b0 + b1) >> 1;
        const float za = a0 < a1 ? quad_z(q, ma) : 0.0f, zb = b0 < b1 ? quad_z(q, mb) : 0.0f;
        if (a0 < a1) {
            if (za < wlo)
                a0 = ma + 1;
            else
                a1 = ma;
        }
        if (b0 < b1) {
            if (zb <= whi)
                b0 = mb + 1;
            else
                b1 = mb;
        }
    }
    lo = a0;
    hi = b0;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Copy bytes (a multiple of 16, both sides aligned to 16) to shared memory, one
// 16-byte unit per lane and round.
__device__ __forceinline__ void warp_copy(uint32_t dst, const void *src, int bytes, int lane)
{
    for (int u = lane * 16; u < bytes; u += 512)
        cp_async16(dst + u, static_cast<const char *>(src) + u);
}

// Two pieces of secondaries per warp in shared memory: while the warp sweeps
// one, the next (of this window or the one after) is on its way.  A 16-byte
// global load of a value that 16 lanes share occupies the L1's data path four
// times (once per quarter warp), a shared load twice.  A Ring says what a piece
// holds: N secondaries, SLOT bytes, copied by copy(P, dst, j, n, lane).
template <int LEN>
struct RingCoords {  // coordinates, in the quad layout
    static constexpr int N = LEN, SLOT = N * 12, BYTES = 2 * SLOT;
    static __device__ __forceinline__ void copy(const PairParams &P, uint32_t dst, int j, int n, int lane)
    {
        warp_copy(dst, P.B.xyz + 3ll * j, n * 12, lane);
    }
};

using RingXYZ = RingCoords<192>;

// Coordinates, then their residuals (RL) in the quad layout, then weights (W).
// Short pieces: two CTAs with their rows of sums fill an SM's shared memory.
template <bool W, bool RL>
struct RingSums {
    static constexpr int N = RL ? 32 : 64, RES_OFF = N * 12, W_OFF = N * (RL ? 24 : 12),
                         SLOT = W_OFF + (W ? N * 4 : 0), BYTES = 2 * SLOT;
    static __device__ __forceinline__ void copy(const PairParams &P, uint32_t dst, int j, int n, int lane)
    {
        warp_copy(dst, P.B.xyz + 3ll * j, n * 12, lane);
        if (RL)
            warp_copy(dst + RES_OFF, P.B.res + 3ll * j, n * 12, lane);
        if (W)
            warp_copy(dst + W_OFF, P.B.ws + j, n * 4, lane);
    }
};

// The job's byte table by one bulk copy into smem + lut_off, while fill() writes
// what else the CTA needs (the barrier at smem is initialised; its phase parity is
// phase).  False in every thread if the wait gave up.
template <class Fill>
__device__ __forceinline__ bool load_table(const PairParams &P, unsigned char *smem, int lut_off,
                                           unsigned phase, Fill fill)
{
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem);
    if (threadIdx.x == 0) {
        const unsigned bytes = ((unsigned)P.lut_n + 15u) & ~15u;
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(bar, bytes);
        if (!(P.flags & CF_FLAG_DEBUG_STALL) || P.kind != 0 || P.wacc)  // diagnostic stall: never issued
            bulk_g2s(smem + lut_off, P.lut, bytes, bar);
    }
    fill();
    if (__syncthreads_or(!mbar_wait(bar, phase, P.wait_ns))) {
        if (threadIdx.x == 0) {
            atomicOr(P.err, ERR_TIMEOUT);
            mbar_wait(bar, phase, P.wait_ns);  // a late copy lands before the CTA exits
        }
        return false;
    }
    return true;
}

// A chunk's primaries: lane ii of I holds the entries ib + q I + ii.
template <int I, int PP>
struct Chunk {
    float x[PP], y[PP], z[PP];
    float zlo, zhi;  // z range of the real entries
    unsigned vmask;  // bit q: entry q is real (column padding is NaN)
    int col;

    // False if the chunk holds only padding.
    __device__ __forceinline__ bool load(const PairParams &P, int ib, int ii)
    {
        col = __ldg(P.A.chunk_col + ib / (int)COL_PAD);
        int zb = 0;
        vmask = 0;
#pragma unroll
        for (int q = 0; q < PP; ++q) {
            const float *p = P.A.xyz + quad_off((uint32_t)(ib + q * I + ii));
            x[q] = __ldg(p);
            y[q] = __ldg(p + 4);
            z[q] = __ldg(p + 8);
            const bool v = !isnan(x[q]);
            vmask |= (unsigned)v << q;
            if (v)  // frame coordinates are >= 0: they order like their bits (-0 below)
                zb = max(zb, __float_as_int(z[q]));
        }
        zlo = __shfl_sync(FULL, z[0], 0);
        zhi = __int_as_float(__reduce_max_sync(FULL, zb));
        return !isnan(zlo);
    }

    // The primaries shifted for image code / k, broadcast into packed pairs;
    // returns the image (qx + 1, qy + 1, qz + 1 in two bits each).
    __device__ __forceinline__ int shift(const PairParams &P, int k, int code, u64 (&XH)[PP], u64 (&YH)[PP],
                                         u64 (&ZH)[PP]) const
    {
        const float Sx = (float)((code & 3) - 1) * P.boxf[0];
        const float Sy = (float)(((code >> 2) & 3) - 1) * P.boxf[1], Sz = (float)k * P.boxf[2];
#pragma unroll
        for (int q = 0; q < PP; ++q) {
            const float xh = __fsub_rn(x[q], Sx), yh = __fsub_rn(y[q], Sy), zh = __fsub_rn(z[q], Sz);
            XH[q] = pack2(xh, xh);
            YH[q] = pack2(yh, yh);
            ZH[q] = pack2(zh, zh);
        }
        return (code & 15) | ((k + 1) << 4);
    }
};

// The windows of the chunk [ib, ib + CH) of column col against its neighbours
// part, part + parts, ...; all lanes call it together.  SL: parts is a multiple of
// nstencil, a part one neighbour (or all, parts 1) and one of parts / nstencil slices
// of its windows.  For every window,
// open(k, code) sets the primaries up for the image, then for every piece
// [j0, j1) of it (j0 a multiple of JS; secondaries outside the window are
// farther than the reach in z) sweep(addr, j0, j1, jlo, jhi, tri) is called with
// the shared address of secondary j0.
template <int JS, class Ring, bool SL, class Open, class Sw>
__device__ __forceinline__ void for_windows(const PairParams &P, int col, int ib, float zlo, float zhi,
                                            int part, int parts, int lane, uint32_t ring, Open open, Sw sw)
{
    const int nn = (int)__ldg(P.nbr_count + col), nz = P.g.nz;
    const Nbr *nb = P.nbr + (long long)col * P.nstencil;
    const int slices = SL && parts > 1 ? parts / P.nstencil : 1, slice = SL ? part % slices : 0;
    if (SL) {
        part /= slices;
        parts /= slices;
    }
    const int k0 = P.g.periodic ? -1 : 0, k1 = P.g.periodic ? 1 : 0;
    for (int base = part; base < nn; base += 32 * parts) {
        const int e = base + lane * parts;
        int code = 0;
        float dz = 0.0f;
        if (e < nn) {
            const int2 r = __ldg(reinterpret_cast<const int2 *>(nb + e));
            dz = __int_as_float(r.x);
            code = r.y;
        }
#pragma unroll 1
        for (int k = k0; k <= k1; ++k) {
            const float kz = (float)k * P.boxf[2];
            const float wlo = zlo - kz - dz, whi = zhi - kz + dz;
            int jlo = 0, jhi = 0;
            // in a periodic box z lies in [0, L), and a self pair takes only one
            // of the images -1 and +1
            if (e < nn && !(P.g.periodic && (whi < 0.0f || wlo > P.boxf[2] || ((code & 16) && k < 0)))) {
                const uint32_t *cs = P.B.cell_start + (long long)(code >> 5) * nz;
                zwindow(P.B.xyz, cs, nz, P.g.inv_wf[2], wlo, whi, jlo, jhi);
                if ((code & 16) && k == 0)
                    jlo = max(jlo, ib + 1);
                if (SL && jlo < jhi) {  // whole steps: a sweep takes all that its steps hold
                    const int s0 = jlo / JS, n = (jhi - 1) / JS + 1 - s0, per = (n + slices - 1) / slices;
                    const int a = min(n, per * slice), b = min(n, a + per);
                    jlo = max(jlo, (s0 + a) * JS);
                    jhi = min(jhi, (s0 + b) * JS);
                }
            }
            unsigned m = __ballot_sync(FULL, jlo < jhi), pm = m;
            if (!m)
                continue;
            int pj = 0, pe = 0;  // the next piece to request: [pj, ...) of the window ending at pe
            auto request = [&](uint32_t dst) {
                if (pj >= pe && pm) {
                    const int l = __ffs(pm) - 1;
                    pm &= pm - 1u;
                    pj = __shfl_sync(FULL, jlo, l) & ~(JS - 1);
                    pe = __shfl_sync(FULL, jhi, l);
                }
                if (pj < pe) {
                    const int n = min(Ring::N, (pe - pj + JS - 1) & ~(JS - 1));
                    Ring::copy(P, dst, pj, n, lane);
                    pj += n;
                }
                cp_commit();
            };
            uint32_t cur = ring;
            request(cur);
            for (; m; m &= m - 1u) {
                const int l = __ffs(m) - 1;
                const int lo = __shfl_sync(FULL, jlo, l), hi = __shfl_sync(FULL, jhi, l);
                const int cd = __shfl_sync(FULL, code, l);
                const bool tri = (cd & 16) && k == 0;
                open(k, cd);
                for (int j0 = lo & ~(JS - 1); j0 < hi; j0 += Ring::N) {
                    request(2 * ring + Ring::SLOT - cur);
                    cp_wait<1>();
                    __syncwarp();
                    sw(cur, j0, min(j0 + Ring::N, hi), lo, hi, tri);
                    __syncwarp();
                    cur = 2 * ring + Ring::SLOT - cur;
                }
            }
        }
    }
}

// Queue the pairs of a piece [j0, j1) of a window [jlo, jhi) that the float32 bounds
// do not prove out of reach (set_cull): KIND 0 by r^2, KIND 1 by rp^2 and |dz|.
// drain() is called whenever pairs were added and leaves room for 32 more.
template <int KIND, int I, int PP, bool EVALS, class Queue, class Drain>
__device__ __forceinline__ void cull_piece(const PairParams &P, Queue *fq, int &qn, u64 &n_eval,
                                           uint32_t addr, int j0, int j1, int jlo, int jhi, bool tri, int jj,
                                           int ii, const u64 (&XH)[PP], const u64 (&YH)[PP],
                                           const u64 (&ZH)[PP], int ib, int image, unsigned vmask, Drain drain)
{
    constexpr int JS = 128 / I;
    const u64 CULL = pack2(-P.cull, -P.cull), ZCULL = pack2(-P.zcull, -P.zcull);
    const uint32_t p0 = addr + 48u * jj;
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
            ulonglong2 vx, vy, vz;
            lds128<0>(p, vx);
            lds128<16>(p, vy);
            lds128<32>(p, vz);
#pragma unroll
            for (int q = 0; q < PP; ++q) {
                u64 s[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const u64 dx = fsub2(h ? vx.y : vx.x, XH[q]), dy = fsub2(h ? vy.y : vy.x, YH[q]),
                              dz = fsub2(h ? vz.y : vz.x, ZH[q]);
                    // negative: within reach (a NaN of the padding is positive)
                    s[h] = ffma2(dy, dy, ffma2(dx, dx, CULL));
                    if (KIND == 0)
                        s[h] = ffma2(dz, dz, s[h]);
                    else  // both signs set
                        s[h] &= ffma2(dz, dz, ZCULL);
                }
                float f[4];
                unpack2(s[0], f[0], f[1]);
                unpack2(s[1], f[2], f[3]);
#pragma unroll
                for (int r = 0; r < 4; ++r)  // pair (t, r) ends at bit 4 tend - 1 - (4 t + r)
                    fm[q] = push_sign(fm[q], __float_as_uint(f[r]));
            }
            if (EVALS) {
                const int jt = j0 + 4 * jj + (int)((p - p0) / 12u);
#pragma unroll
                for (int q = 0; q < PP; ++q)
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        n_eval += (((vmask >> q) & 1u) && jt + r >= jlo && jt + r < jhi &&
                                   (!tri || jt + r > ib + q * I + ii)) ? 1ull : 0ull;
            }
        }
        const int lane = threadIdx.x & 31, jb = j0 + 4 * jj + (int)((pb - p0) / 12u);
#pragma unroll
        for (int q = 0; q < PP; ++q) {
            const int i = ib + q * I + ii;
            uint32_t m = fm[q];
            for (unsigned bm; (bm = __ballot_sync(FULL, m != 0u)) != 0u;) {
                const int b = 4 * tend - __ffs(m);  // = 4 t + r
                const int j = jb + (b >> 2) * JS + (b & 3);
                const bool put = m != 0u && (!tri || j > i);
                m &= m - 1u;
                if (tri)
                    bm = __ballot_sync(FULL, put);
                if (put) {
                    const int at = qn + __popc(bm & ((1u << lane) - 1u));
                    fq->i[at] = i;
                    fq->j[at] = j;
                    fq->image[at] = image;
                }
                qn += __popc(bm);
                drain();
            }
        }
    }
}

// Neighbour lists (Sec. 2.1, 2.2): one warp per primary column, one stencil
// offset per lane; the kept column pairs are listed in stencil order with
// their z reach (float32, rounded up, with the window slack).
__device__ __forceinline__ void neighbours_body(const PairParams &P, int col, int lane)
{
    if (col >= P.g.ncols)
        return;
    int n = 0;
    for (int s0 = 0; s0 < P.nstencil; s0 += 32) {
        const int s = s0 + lane;
        Nbr r;
        const bool keep = s < P.nstencil && plan_item(P, col * P.nstencil + s, r);
        const unsigned m = __ballot_sync(FULL, keep);
        if (keep)
            P.nbr[(long long)col * P.nstencil + n + __popc(m & ((1u << lane) - 1u))] = r;
        n += __popc(m);
    }
    if (lane == 0) {
        P.nbr_count[col] = (unsigned)n;
        if (n)
            atomicAdd(P.work_count, (unsigned)n);
    }
}

// Warps per CTA of a path: Path::NW, or WARPS.
template <class Path>
constexpr auto path_warps_of(int) -> decltype(Path::NW)
{
    return Path::NW;
}
template <class Path>
constexpr int path_warps_of(long)
{
    return WARPS;
}
template <class Path>
constexpr int path_warps()
{
    return path_warps_of<Path>(0);
}

// Persistent kernel over the chunk tasks of one count.  Path: CH (primaries per
// chunk), State, init (false in every thread if the CTA has to give up), task,
// fini.
template <class Path, int MINB>
__global__ void __launch_bounds__(32 * path_warps<Path>(), MINB) k_tasks(const __grid_constant__ PairParams P)
{
    extern __shared__ __align__(128) unsigned char smem[];
    typename Path::State st;
    if (!Path::init(P, smem, st))
        return;
    const int lane = threadIdx.x & 31;
    const unsigned nchunk = __ldg(P.A.cell_start + P.g.ncells) / Path::CH;
    const TaskSplit split(nchunk, (unsigned)P.parts, nchunk <= 2u * gridDim.x * path_warps<Path>());
    unsigned nxt = 0;
    if (lane == 0)
        nxt = atomicAdd(P.item_counter, 1u);
    for (unsigned t = __shfl_sync(FULL, nxt, 0); t < split.ntask; t = __shfl_sync(FULL, nxt, 0)) {
        if (lane == 0)
            nxt = atomicAdd(P.item_counter, 1u);  // read at the end of this task
        unsigned c, part, parts;
        split.task(t, c, part, parts);
        Path::task(P, smem, st, c, part, parts);
    }
    Path::fini(P, smem, st);
}

// Launch k_tasks with L.smem bytes of shared memory per CTA; Sliced: the path's variant for
// sliced windows (SL), if it has one.
template <class Path, int MINB, class Sliced = Path>
cudaError_t launch_tasks(const PairParams &P0, PairLaunch &L, int sms, cudaStream_t st)
{
    PairParams P = P0;
    int occ = 0;
    constexpr int NW = path_warps<Path>();
    const cudaError_t e = occupancy(k_tasks<Path, MINB>, L.smem, occ, 32 * NW);
    if (e)
        return e;
    if (occ < 1)
        return cudaErrorInvalidConfiguration;
    const long long chunks = (P.A.n + (long long)P.g.ncols * (COL_PAD / 2)) / Path::CH + 1;
    P.parts = task_parts((double)chunks, (double)sms * occ * NW, P.nstencil);
    if (!std::is_same<Path, Sliced>::value) {
        const int slices = task_slices((double)chunks, (double)sms * occ * NW, P.nstencil, window_points(P, Path::CH));
        if (slices > 1) {
            P.parts = P.nstencil * slices;
            const cudaError_t es = occupancy(k_tasks<Sliced, MINB>, L.smem, occ, 32 * NW);
            if (es)
                return es;
            if (occ < 1)
                return cudaErrorInvalidConfiguration;
            L.blocks = (int)std::min<long long>((long long)sms * occ, (chunks * P.parts + NW - 1) / NW);
            k_tasks<Sliced, MINB><<<L.blocks, 32 * NW, L.smem, st>>>(P);
            return cudaGetLastError();
        }
    }
    L.blocks = (int)std::max(1ll, std::min<long long>((long long)sms * occ, (chunks * P.parts + NW - 1) / NW));
    k_tasks<Path, MINB><<<L.blocks, 32 * NW, L.smem, st>>>(P);
    return cudaGetLastError();
}

}  // namespace

}  // namespace cf
