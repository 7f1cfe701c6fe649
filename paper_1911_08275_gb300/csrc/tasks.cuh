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

// Two pieces of secondaries per warp in shared memory: while the warp sweeps
// one, the next (of this window or the one after) is on its way.  A 16-byte
// global load of a value that 16 lanes share occupies the L1's data path four
// times (once per quarter warp), a shared load twice.
constexpr int PIECE = 192;                   // secondaries per piece
constexpr int PIECE_BYTES = PIECE * 12;      // in the quad layout
constexpr int RING_BYTES = 2 * PIECE_BYTES;  // per warp

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
        if (!(P.flags & CF_FLAG_DEBUG_STALL) || P.kind != 0)  // diagnostic stall: never issued
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
// part, part + parts, ...; all lanes call it together.  For every window,
// open(k, code) sets the primaries up for the image, then for every piece
// [j0, j1) of it (j0 a multiple of JS; secondaries outside the window are
// farther than the reach in z) sweep(addr, j0, j1, jlo, jhi, tri) is called with
// the shared address of secondary j0.
template <int JS, class Open, class Sw>
__device__ __forceinline__ void for_windows(const PairParams &P, int col, int ib, float zlo, float zhi,
                                            int part, int parts, int lane, uint32_t ring, Open open, Sw sw)
{
    const int nn = (int)__ldg(P.nbr_count + col), nz = P.g.nz;
    const Nbr *nb = P.nbr + (long long)col * P.nstencil;
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
                    const int n = min(PIECE, (pe - pj + JS - 1) & ~(JS - 1));
                    const char *src = reinterpret_cast<const char *>(P.B.xyz) + 12ll * pj;
                    for (int u = lane * 16; u < n * 12; u += 512)
                        cp_async16(dst + u, src + u);
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
                for (int j0 = lo & ~(JS - 1); j0 < hi; j0 += PIECE) {
                    request(2 * ring + PIECE_BYTES - cur);
                    cp_wait<1>();
                    __syncwarp();
                    sw(cur, j0, min(j0 + PIECE, hi), lo, hi, tri);
                    __syncwarp();
                    cur = 2 * ring + PIECE_BYTES - cur;
                }
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
        WorkItem w;
        const bool keep = s < P.nstencil && plan_item(P, col * P.nstencil + s, w);
        const unsigned m = __ballot_sync(FULL, keep);
        if (keep) {
            Nbr r;
            r.dz = __fadd_ru(__double2float_ru(w.dzmax), P.zslack);
            r.code = w.code;
            P.nbr[(long long)col * P.nstencil + n + __popc(m & ((1u << lane) - 1u))] = r;
        }
        n += __popc(m);
    }
    if (lane == 0) {
        P.nbr_count[col] = (unsigned)n;
        if (n)
            atomicAdd(P.work_count, (unsigned)n);
    }
}

// Persistent kernel over the chunk tasks of one count.  Path: CH (primaries per
// chunk), State, init (false in every thread if the CTA has to give up), task,
// fini.
template <class Path, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) k_tasks(const __grid_constant__ PairParams P)
{
    extern __shared__ __align__(128) unsigned char smem[];
    typename Path::State st;
    if (!Path::init(P, smem, st))
        return;
    const int lane = threadIdx.x & 31;
    const unsigned nchunk = __ldg(P.A.cell_start + P.g.ncells) / Path::CH;
    const TaskSplit split(nchunk, (unsigned)P.parts, nchunk <= 2u * gridDim.x * WARPS);
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

// Launch k_tasks with L.smem bytes of shared memory per CTA.
template <class Path, int MINB>
cudaError_t launch_tasks(const PairParams &P0, PairLaunch &L, int sms, cudaStream_t st)
{
    PairParams P = P0;
    int occ = 0;
    const cudaError_t e = occupancy(k_tasks<Path, MINB>, L.smem, occ);
    if (e)
        return e;
    if (occ < 1)
        return cudaErrorInvalidConfiguration;
    const long long chunks = (P.A.n + (long long)P.g.ncols * (COL_PAD / 2)) / Path::CH + 1;
    P.parts = task_parts((double)chunks, (double)sms * occ * WARPS, P.nstencil);
    L.blocks = (int)std::max(1ll, std::min<long long>((long long)sms * occ, (chunks * P.parts + WARPS - 1) / WARPS));
    k_tasks<Path, MINB><<<L.blocks, THREADS, L.smem, st>>>(P);
    return cudaGetLastError();
}

}  // namespace

}  // namespace cf
