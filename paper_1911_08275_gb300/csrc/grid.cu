// GPU gridding (Sec. 1.2 and 2.1 of arXiv:1911.08275): points are binned into
// columns of side >= Rmax / refine in x and y, each column is sorted along z
// (the paper's z-sort that shrinks the search window from 3*pimax to 2*pimax),
// and each column gets its (x, y) bounding box for the pruning of Sec. 2.2.
//
// Layout produced (one gridded catalogue):
//   cell_start[ncells + 1]  counting-sort offsets; cell = column * nz + zcell,
//                           column = cx * ncy + cy.  A column is the contiguous
//                           range [cell_start[col*nz], cell_start[(col+1)*nz]),
//                           padded at its end to a multiple of COL_PAD = 32
//                           entries, so chunks of 8, 16 or 32 primaries and
//                           aligned groups of secondaries never straddle two
//                           columns; padding entries are NaN and never counted.
//   xyz[3 n']       float32 x - ox, y - oy, z - oz (grid frame) in quads (x0..x3, y0..y3,
//                   z0..z3 per four points)
//   chunk_col[n'/32] column of each run of 32 entries
//   pos64[n']       double4 (x, y, z, w) exact binary64 copies (re-checks, FP64 path)
//   perm[n']        original index of each sorted point (-1 for padding)
//   colbox[ncols]   (xmin, xmax, ymin, ymax) of the column's points, binary64
// with n' <= n + 31 * ncols.
//
// Within a cell the order is (z, original index), computed by ranking, so the
// output is deterministic whatever the order of the atomic slot assignment.
#include <cuda_runtime.h>
#include <float.h>

#include <algorithm>
#include <mutex>

#include "cf_internal.cuh"
#include "grid.cuh"
#include "launch.cuh"

namespace cf {

namespace {

// Unique id of the calling thread's current CUDA context (cuCtxGetId, reached
// through the runtime's driver entry points so the library does not link the
// driver library).  A device reset or a new context gets a new id.
typedef int (*PfnCtxGetCurrent)(void **);
typedef int (*PfnCtxGetId)(void *, unsigned long long *);

}  // namespace

bool current_context_id(int dev, unsigned long long &id)
{
    static PfnCtxGetCurrent get_current = nullptr;
    static PfnCtxGetId get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, []() {
        cudaDriverEntryPointQueryResult q1, q2;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", (void **)&get_current, 12000,
                                             cudaEnableDefault, &q1) != cudaSuccess ||
            q1 != cudaDriverEntryPointSuccess)
            get_current = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", (void **)&get_id, 12000,
                                             cudaEnableDefault, &q2) != cudaSuccess ||
            q2 != cudaDriverEntryPointSuccess)
            get_id = nullptr;
        cudaGetLastError();
    });
    if (!get_current || !get_id)
        return false;
    void *ctx = nullptr;
    if (get_current(&ctx) != 0 || !ctx) {
        // no current context yet: make the device's primary context current
        if (cudaSetDevice(dev) != cudaSuccess || get_current(&ctx) != 0 || !ctx) {
            cudaGetLastError();
            return false;
        }
    }
    return get_id(ctx, &id) == 0;
}

namespace {

// Binary64 -> float32, round to nearest even, and back, in integer arithmetic: the
// conversion instructions run in the binary64 pipe, two lanes per SM (gridding
// 1.2M points held it busy for half of the time).  Zeros are taken as they are;
// values whose float32 is not a normal number take the instruction.
__device__ __forceinline__ float d2f(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned e = (unsigned)(b >> 52) & 0x7ffu;
    if (e - 897u < 253u) {  // 2^-126 <= |v| < 2^127
        const unsigned long long r = b + 0x0fffffffull + ((b >> 29) & 1ull);
        return __uint_as_float((((unsigned)(r >> 29) - (896u << 23)) & 0x7fffffffu) |
                               ((unsigned)(b >> 32) & 0x80000000u));
    }
    if ((b << 1) == 0ull)
        return __uint_as_float((unsigned)(b >> 32));
    return __double2float_rn(v);
}
__device__ __forceinline__ double f2d(float v)
{
    const unsigned u = __float_as_uint(v);
    if (((u >> 23) & 0xffu) - 1u < 254u)
        return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))),
                                (int)(u << 29));
    if ((u << 1) == 0u)
        return __hiloint2double((int)u, 0);
    return (double)v;
}
__device__ __forceinline__ double to_f64(double v) { return v; }
__device__ __forceinline__ double to_f64(float v) { return f2d(v); }

// Validity and float32 frame coordinate of one input coordinate, without
// binary64 arithmetic in a periodic box (the binary64 pipe of this GPU is narrow):
// range tests on bit patterns.
__device__ __forceinline__ bool coord(double v, int a, const Geom &g, float &f)
{
    const long long b = __double_as_longlong(v);
    if (g.periodic) {
        f = d2f(v);  // frame origin is 0
        return (b >= 0 && b < g.box_bits[a]) || b == (long long)0x8000000000000000ull;
    }
    f = d2f(__dsub_rn(v, g.origin[a]));
    return (b & 0x7ff0000000000000ll) != 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool coord(float v, int a, const Geom &g, float &f)
{
    const int b = __float_as_int(v);
    if (g.periodic) {
        f = v;
        return (b >= 0 && b < g.box_bits32[a]) || b == (int)0x80000000u;
    }
    f = d2f(__dsub_rn(f2d(v), g.origin[a]));
    return (b & 0x7f800000) != 0x7f800000;
}

// Sum over the block (every thread gets it; red: one word per warp).
__device__ __forceinline__ uint32_t block_sum(uint32_t v, uint32_t *red)
{
    v = __reduce_add_sync(FULL, v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0)
        red[threadIdx.x >> 5] = v;
    __syncthreads();
    uint32_t s = 0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q)
        s += red[q];
    return s;
}

// Cell and slot in the cell of every point (counts of the cells in count, zeroed).
template <class T>
__device__ __forceinline__ void assign_points(const T *__restrict__ x, const T *__restrict__ y,
                                              const T *__restrict__ z, long long n, const Geom &g,
                                              uint32_t *cell_of, uint32_t *slot, uint32_t *count, unsigned *err,
                                              unsigned blk, unsigned nblk)
{
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)nblk * blockDim.x;
    // every lane of a warp runs the same number of iterations (warp-wide match)
    const long long first = (long long)blk * blockDim.x + (threadIdx.x & ~31);
    for (long long base = first; base < n; base += stride) {
        const long long p = base + lane;
        const bool live = p < n;
        uint32_t cell = 0xffffffffu;
        if (live) {
            float fx, fy, fz;
            const bool ok = coord(x[p], 0, g, fx) & coord(y[p], 1, g, fy) & coord(z[p], 2, g, fz);
            if (!ok) {
                atomicOr(err, ERR_COORD);
                fx = fy = fz = 0.0f;
            }
            const int cx = cell_index_f(fx, g.inv_wf[0], g.ncx);
            const int cy = cell_index_f(fy, g.inv_wf[1], g.ncy);
            const int cz = cell_index_f(fz, g.inv_wf[2], g.nz);
            cell = (uint32_t)(((long long)(cx * g.ncy + cy)) * g.nz + cz);
        }
        // clustered inputs put runs of points into one cell: one atomic per group
        const unsigned same = __match_any_sync(FULL, cell);
        const int leader = __ffs(same) - 1;
        uint32_t b0 = 0;
        if (live && lane == leader)
            b0 = atomicAdd(&count[cell], (uint32_t)__popc(same));
        b0 = __shfl_sync(FULL, b0, leader);
        if (live) {
            cell_of[p] = cell;
            slot[p] = b0 + (uint32_t)__popc(same & ((1u << lane) - 1u));
        }
    }
}

// Exclusive scan, 3 phases: per-block scan of SCAN_ITEMS elements, scan of the
// block sums (one block), add-back.
constexpr int SCAN_THREADS = 1024;
constexpr int SCAN_PER_THREAD = 4;
constexpr int SCAN_ITEMS = SCAN_THREADS * SCAN_PER_THREAD;

__device__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *warp_sums, uint32_t *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(FULL, incl, o);
        if (lane >= o)
            incl += t;
    }
    if (lane == 31)
        warp_sums[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        const int nw = blockDim.x >> 5;
        uint32_t s = lane < nw ? warp_sums[lane] : 0u;
        uint32_t si = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t t = __shfl_up_sync(FULL, si, o);
            if (lane >= o)
                si += t;
        }
        if (lane < nw)
            warp_sums[lane] = si - s;
        if (lane == 31)
            *total = si;
    }
    __syncthreads();
    const uint32_t r = warp_sums[wid] + incl - v;
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(SCAN_THREADS)
    k_scan_blocks(const uint32_t *in, uint32_t *out, long long n, uint32_t *__restrict__ bsum)
{
    __shared__ uint32_t ws[32];
    __shared__ uint32_t tot;
    const long long base = (long long)blockIdx.x * SCAN_ITEMS + threadIdx.x * SCAN_PER_THREAD;
    uint32_t v[SCAN_PER_THREAD];
    uint32_t s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_PER_THREAD; ++k) {
        v[k] = (base + k < n) ? in[base + k] : 0u;
        s += v[k];
    }
    uint32_t pre = block_exclusive_scan(s, ws, &tot);
#pragma unroll
    for (int k = 0; k < SCAN_PER_THREAD; ++k) {
        if (base + k < n)
            out[base + k] = pre;
        pre += v[k];
    }
    if (threadIdx.x == 0)
        bsum[blockIdx.x] = tot;
}

// Exclusive scan of the block sums in place (one block, SCAN_ITEMS at a time
// with a running carry); *grand gets the total.
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_sums(uint32_t *bsum, long long nb, uint32_t *grand)
{
    __shared__ uint32_t ws[32];
    __shared__ uint32_t tot;
    uint32_t carry = 0;
    for (long long c = 0; c < nb; c += SCAN_ITEMS) {
        uint32_t v[SCAN_PER_THREAD];
        uint32_t s = 0;
        const long long base = c + threadIdx.x * SCAN_PER_THREAD;
#pragma unroll
        for (int k = 0; k < SCAN_PER_THREAD; ++k) {
            v[k] = (base + k < nb) ? bsum[base + k] : 0u;
            s += v[k];
        }
        uint32_t pre = carry + block_exclusive_scan(s, ws, &tot);
#pragma unroll
        for (int k = 0; k < SCAN_PER_THREAD; ++k) {
            if (base + k < nb)
                bsum[base + k] = pre;
            pre += v[k];
        }
        carry += tot;  // read before any thread can reach the next scan's write of tot
    }
    if (threadIdx.x == 0)
        *grand = carry;
}

__global__ void k_scan_add(uint32_t *__restrict__ out, long long n, const uint32_t *__restrict__ bsum)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n)
        out[i] += bsum[i / SCAN_ITEMS];
}

// Write one ranked entry: binary64 copy, float32 frame coordinates, their rounding
// residuals fl32((X - O) - x~) if wanted, weight, original index.
template <class T>
__device__ __forceinline__ void put_entry(const T *__restrict__ x, const T *__restrict__ y,
                                          const double *__restrict__ w, const Geom &g, uint32_t d,
                                          int iq, unsigned long long kq, const Gridded &G, unsigned &wm,
                                          ColBox &box)
{
    const double X = to_f64(x[iq]), Y = to_f64(y[iq]), Z = key_value(kq);
    const unsigned long long kx = order_key(__double_as_longlong(X)), ky = order_key(__double_as_longlong(Y));
    box.x0 = min(box.x0, kx);
    box.x1 = max(box.x1, kx);
    box.y0 = min(box.y0, ky);
    box.y1 = max(box.y1, ky);
    const double W = w ? w[iq] : 0.0;
    G.pos64[d] = make_double4_32a(X, Y, Z, W);
    const double fx = g.periodic ? X : __dsub_rn(X, g.origin[0]);
    const double fy = g.periodic ? Y : __dsub_rn(Y, g.origin[1]);
    const double fz = g.periodic ? Z : __dsub_rn(Z, g.origin[2]);
    const float sx = d2f(fx), sy = d2f(fy), sz = d2f(fz);
    float *qd = G.xyz + quad_off(d);
    qd[0] = sx;
    qd[4] = sy;
    qd[8] = sz;
    if (G.res) {  // float32 mean separations restore the coordinates' lost bits
        float *rd = G.res + quad_off(d);
        rd[0] = d2f(__dsub_rn(fx, f2d(sx)));
        rd[4] = d2f(__dsub_rn(fy, f2d(sy)));
        rd[8] = d2f(__dsub_rn(fz, f2d(sz)));
    }
    if (G.ws) {
        const float wf = d2f(W);
        G.ws[d] = wf;
        wm = max(wm, __float_as_uint(fabsf(wf)));
    }
    G.perm[d] = iq;
}

constexpr int SORT_THREADS = 256;
constexpr int SORT_BUF = 256;  // entries of a cell ranked from shared memory

// Rank of entry (kq, iq) among the n entries of e[] by (key, original index).
__device__ __forceinline__ uint32_t rank_in(const ulonglong2 *e, uint32_t n, unsigned long long kq,
                                            int iq)
{
    uint32_t rank = 0;
    for (uint32_t m = 0; m < n; ++m) {
        const ulonglong2 em = e[m];  // every lane of the group reads the same entry
        rank += (em.x < kq) || (em.x == kq && (int)em.y < iq);
    }
    return rank;
}

__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v)
{
    const unsigned hi = __reduce_min_sync(FULL, (unsigned)(v >> 32));
    const unsigned lo = __reduce_min_sync(FULL, (unsigned)(v >> 32) == hi ? (unsigned)v : ~0u);
    return ((unsigned long long)hi << 32) | lo;
}
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) { return ~warp_min_u64(~v); }

__device__ __forceinline__ ColBox empty_box() { return ColBox{~0ull, 0ull, ~0ull, 0ull}; }

// Rank the real entries of a warp's cells by (z, original index) and write the
// sorted outputs; lane l holds cell l of a run of consecutive cells (count n,
// offset s, column col; n = 0 past the run's end).  Cells are ordered by z within a
// column, so neighbouring cells of one column that hold at most 32 entries
// together are ranked as one group, one entry per lane; a larger cell by itself,
// from the warp's buffer up to SORT_BUF entries, beyond that in global memory.  The
// entries being ranked are 16-byte (key, index) records: one broadcast load per
// comparison.  at(l, col): the arrays of lane l's cell and the box of its column (all
// lanes call it); put(src, d, iq, kq, box): write entry d.
template <class At, class Put>
__device__ __forceinline__ void sort_run(uint32_t n, uint32_t s, int col, int lane, ulonglong2 *be, At at,
                                         Put put)
{
    uint32_t incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(FULL, incl, o);
        if (lane >= o)
            incl += t;
    }
    for (unsigned todo = __ballot_sync(FULL, n > 0u); todo;) {
        const int k = __ffs(todo) - 1;
        const uint32_t before = __shfl_sync(FULL, incl - n, k), nk = __shfl_sync(FULL, n, k);
        const uint32_t sk = __shfl_sync(FULL, s, k);
        const int ck = __shfl_sync(FULL, col, k);
        unsigned grp = __ballot_sync(FULL, n > 0u && lane >= k && col == ck && incl - before <= 32u);
        if (nk > 32u)
            grp = 1u << k;
        const uint32_t cn = __shfl_sync(FULL, incl, 31 - __clz(grp)) - before;  // entries of the group
        todo &= ~grp;
        const auto src = at(k, ck);
        ColBox box = empty_box();
        const bool buffered = cn <= (uint32_t)SORT_BUF;
        if (buffered) {
            __syncwarp();
            for (uint32_t e = lane; e < cn; e += 32)
                be[e] = make_ulonglong2(src.key[sk + e], (unsigned long long)(unsigned)src.idx[sk + e]);
            __syncwarp();
        }
        for (uint32_t e0 = 0; e0 < cn; e0 += 32) {
            const uint32_t e = e0 + lane;
            if (e < cn) {
                unsigned long long kq;
                int iq;
                uint32_t rank = 0;
                if (buffered) {
                    kq = be[e].x;
                    iq = (int)be[e].y;
                    rank = rank_in(be, cn, kq, iq);
                } else {
                    kq = src.key[sk + e];
                    iq = src.idx[sk + e];
                    for (uint32_t m = 0; m < cn; ++m) {
                        const unsigned long long km = src.key[sk + m];
                        const int im = src.idx[sk + m];
                        rank += (km < kq) || (km == kq && im < iq);
                    }
                }
                put(src, sk + rank, iq, kq, box);
            }
        }
        __syncwarp();
        box.x0 = warp_min_u64(box.x0);
        box.x1 = warp_max_u64(box.x1);
        box.y0 = warp_min_u64(box.y0);
        box.y1 = warp_max_u64(box.y1);
        if (lane == 0) {
            atomicMin(&src.box->x0, box.x0);
            atomicMax(&src.box->x1, box.x1);
            atomicMin(&src.box->y0, box.y0);
            atomicMax(&src.box->y1, box.y1);
        }
    }
}

struct SortSrc {
    const unsigned long long *key;
    const int *idx;
    ColBox *box;
};
struct SegSrc : SortSrc {
    const GridSeg *seg;
};

// Cells of one claim: enough claims for four per warp, up to 32 cells.
__device__ __forceinline__ unsigned claim_cells(long long ncells)
{
    const long long per = ncells / (4ll * gridDim.x * (SORT_THREADS / 32));
    return per >= 32 ? 32u : per < 2 ? 2u : (unsigned)per;
}

template <class T>
__device__ __forceinline__ void sort_cells(const T *__restrict__ x, const T *__restrict__ y,
                                           const double *__restrict__ w, long long ncells, const Geom &g,
                                           const uint32_t *count, const int *tmp_idx,
                                           const unsigned long long *tmp_key, const Gridded &G, unsigned *claim,
                                           ulonglong2 (*s_ent)[SORT_BUF])
{
    const uint32_t *start = G.cell_start;  // written earlier in the same launch: plain loads
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned per = claim_cells(ncells);
    unsigned wm = 0;  // bit pattern of the largest |w| (float) this thread stored
    for (;;) {
        unsigned v = 0u;
        if (lane == 0)
            v = atomicAdd(claim, per);  // the next run of cells (zeroed with the counts)
        const long long c = (long long)__shfl_sync(FULL, v, 0) + lane;
        if (c - lane >= ncells)
            break;
        const bool mine = (unsigned)lane < per && c < ncells;
        const uint32_t n = mine ? count[c] : 0u, s = mine ? start[c] : 0u;
        sort_run(n, s, mine ? (int)c / g.nz : -1, lane, s_ent[wid],
                 [&](int, int k) { return SortSrc{tmp_key, tmp_idx, G.colbox + k}; },
                 [&](const SortSrc &, uint32_t d, int iq, unsigned long long kq, ColBox &box) {
                     put_entry(x, y, w, g, d, iq, kq, G, wm, box);
                 });
    }
    if (G.ws) {  // one atomic per block
        __shared__ unsigned red[SORT_THREADS / 32];
        wm = __reduce_max_sync(FULL, wm);
        if (lane == 0)
            red[wid] = wm;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned m = 0;
            for (int q = 0; q < SORT_THREADS / 32; ++q)
                m = max(m, red[q]);
            atomicMax(G.wmax, m);
        }
    }
}

// One warp per column: its padding entries (NaN, never counted; perm -1) and
// the column of each of its runs of COL_PAD entries.
__device__ __forceinline__ void pad_column(const Gridded &G, int col, uint32_t s, uint32_t e,
                                           uint32_t pad, int lane)
{
    const float fn = __int_as_float(0x7fc00000);
    const double dn = __longlong_as_double(0x7ff8000000000000ll);
    if ((uint32_t)lane < pad) {
        const uint32_t q = e - 1u - lane;
        float *qd = G.xyz + quad_off(q);
        qd[0] = qd[4] = qd[8] = fn;
        if (G.res) {
            float *rd = G.res + quad_off(q);
            rd[0] = rd[4] = rd[8] = 0.0f;
        }
        if (G.ws)
            G.ws[q] = 0.0f;
        G.pos64[q] = make_double4_32a(dn, dn, dn, dn);
        G.perm[q] = -1;
    }
    for (uint32_t k = s / COL_PAD + lane; k < e / COL_PAD; k += 32)
        G.chunk_col[k] = col;
}

// Everything one catalogue's gridding needs (kernel parameter).
struct GridArgs {
    const void *x, *y, *z;
    const double *w;
    long long n;
    Geom g;
    GridTemps t;
    Gridded out;
    unsigned *err;
    unsigned long long *tickets;  // low half: handed out, high half: finished (zero before the launch)
    int stall;                    // diagnostic: wait for a ticket that does not exist, 1 ms at most
};

// The stages of a launch are split into one ticket per block.  Blocks take the tickets in
// order, a stage's after all of the stage before, and begin one when every ticket of the
// earlier stages is finished: those were taken before it, by blocks that are running, so
// nobody waits for a block that has not started (its place may be held by another
// kernel for any time; the running blocks then take its tickets).

// A block's ticket: share blk of the stage.
struct Ticket {
    unsigned stage, blk;
};

// Finishes the block's ticket (but for the first call) and takes the next, t; false in
// every thread if the wait for the earlier stages gave up (the error word says so; no
// later kernel touches the results).  The limit is 20 s of the GPU's timer and a million
// tries: the timer runs on while another process has the GPU.  One atomic finishes and
// takes: two words cost 1 us more per stage.
__device__ __forceinline__ bool next_ticket(const GridArgs &A, bool first, Ticket &t)
{
    __shared__ Ticket s_t;
    bool ok = true;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        unsigned long long v = atomicAdd(A.tickets, first ? 1ull : (1ull << 32) + 1ull);
        unsigned stage = first ? 0u : t.stage, blk = (unsigned)v - stage * gridDim.x;
        for (; blk >= gridDim.x; blk -= gridDim.x)
            ++stage;
        if (!first)
            v += 1ull << 32;
        const unsigned goal = stage * gridDim.x;  // the tickets of the earlier stages
        uint64_t t0 = 0;
        for (unsigned it = 0; (unsigned)(v >> 32) < goal || (A.stall && goal); ++it) {
            if ((it & 63u) == 63u) {
                const uint64_t now = global_ns();
                t0 = t0 ? t0 : now;
                if (A.stall ? now - t0 > 1000000ull : it >= 1u << 20 && now - t0 > 20000000000ull) {
                    atomicOr(A.err, ERR_TIMEOUT);
                    ok = false;
                    break;
                }
            }
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(A.tickets) : "memory");
        }
        __threadfence();
        s_t = Ticket{stage, blk};
    }
    ok = !__syncthreads_or(!ok);
    t = s_t;
    return ok;
}

// One catalogue's gridding in one launch; its stages:
//   clear the cell counts | cell and slot of every point | padded size of every
//   column, each block over a range of columns | offsets, padding, chunk_col |
//   scatter into cells | rank the cells' entries, write the outputs and column boxes
// Bound: latency (waits of 1.5 us between the stages, dependent loads) for small
// catalogues, the scattered reads of x and y by the ranked order for large ones.  Measured,
// with ten kernels before, one per stage and with conversions in the binary64 pipe: 20,000
// points 36 us of kernels and as much in gaps -> 18 us; 1.2M 113 -> 73 us; 12M
// weighted with residuals 2.2 -> 1.5 ms (k_sort 1,137 -> 850 us by ranking small cells
// together and claiming up to 32 at a time).  A cooperative launch with barriers of the whole
// grid in the place of the tickets took as long (100,000 to 12M points: within 3 us), but two
// of them must not run at once: 40 calls with 300,000 points on each of four streams
// 31.6 ms so, 29.2 ms with tickets.
template <class T>
__global__ void __launch_bounds__(SORT_THREADS) k_grid(const __grid_constant__ GridArgs A)
{
    __shared__ ulonglong2 s_ent[SORT_THREADS / 32][SORT_BUF];
    __shared__ uint32_t s_red[32], s_scan[32], s_tot;
    __shared__ uint32_t s_off[SORT_THREADS];
    const Geom &g = A.g;
    const T *x = (const T *)A.x, *y = (const T *)A.y, *z = (const T *)A.z;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nwarp = SORT_THREADS / 32;
    const unsigned nblk = gridDim.x;
    const long long nc = g.ncells, stride = (long long)nblk * SORT_THREADS;
    uint32_t *counts = A.t.counts, *start = A.out.cell_start;

    Ticket t;
    for (bool begin = true; next_ticket(A, begin, t); begin = false) {
        const unsigned blk = t.blk;
        const long long first = (long long)blk * SORT_THREADS + tid;
        // this ticket's columns (stages 2 and 3)
        const int c0 = (int)((long long)g.ncols * blk / nblk), c1 = (int)((long long)g.ncols * (blk + 1) / nblk);
        switch (t.stage) {
        case 0:
            for (long long q = first; q <= nc; q += stride)  // + the sort's claim counter
                counts[q] = 0u;
            for (long long q = first; q < g.ncols; q += stride)
                A.out.colbox[q] = empty_box();
            break;
        case 1:
            assign_points<T>(x, y, z, A.n, g, A.t.cell_of, A.t.slot, counts, A.err, blk, nblk);
            break;
        case 2: {  // a warp per column adds up its cells
            uint32_t mine = 0;
            for (int col = c0 + wid; col < c1; col += nwarp) {
                uint32_t tot = 0;
                for (int q = lane; q < g.nz; q += 32)
                    tot += counts[(long long)col * g.nz + q];
                tot = __reduce_add_sync(FULL, tot);
                if (lane == 0) {
                    A.t.coltot[col] = tot;
                    mine += (tot + COL_PAD - 1u) & ~(COL_PAD - 1u);
                }
            }
            mine = block_sum(lane == 0 ? mine : 0u, s_red);
            if (tid == 0)
                A.t.bsum[blk] = mine;
            break;
        }
        case 3: {
            uint32_t base = 0;
            for (unsigned q = tid; q < blk; q += SORT_THREADS)
                base += __ldcg(A.t.bsum + q);
            base = block_sum(base, s_red);
            for (int r0 = c0; r0 < c1; r0 += SORT_THREADS) {
                const int col = r0 + tid;
                const uint32_t tot = col < c1 ? A.t.coltot[col] : 0u;
                s_off[tid] = base + block_exclusive_scan((tot + COL_PAD - 1u) & ~(COL_PAD - 1u), s_scan, &s_tot);
                __syncthreads();
                for (int k = wid; k < min(SORT_THREADS, c1 - r0); k += nwarp) {
                    uint32_t off = s_off[k];
                    const uint32_t s = off;
                    const long long cell = (long long)(r0 + k) * g.nz;
                    // four loads in flight: few columns have many cells each (2M points, 49 columns:
                    // the whole gridding 380 -> 339 us)
                    for (int q0 = 0; q0 < g.nz; q0 += 128) {
                        uint32_t v[4];
#pragma unroll
                        for (int h = 0; h < 4; ++h)
                            v[h] = q0 + 32 * h + lane < g.nz ? counts[cell + q0 + 32 * h + lane] : 0u;
#pragma unroll
                        for (int h = 0; h < 4; ++h) {
                            if (q0 + 32 * h >= g.nz)
                                break;
                            uint32_t incl = v[h];
#pragma unroll
                            for (int o = 1; o < 32; o <<= 1) {
                                const uint32_t u = __shfl_up_sync(FULL, incl, o);
                                if (lane >= o)
                                    incl += u;
                            }
                            if (q0 + 32 * h + lane < g.nz)
                                start[cell + q0 + 32 * h + lane] = off + incl - v[h];
                            off += __shfl_sync(FULL, incl, 31);
                        }
                    }
                    const uint32_t e = s + ((off - s + COL_PAD - 1u) & ~(COL_PAD - 1u));
                    pad_column(A.out, r0 + k, s, e, e - off, lane);
                    if (r0 + k == g.ncols - 1 && lane == 0)
                        start[nc] = e;
                }
                base += s_tot;
                __syncthreads();
            }
            break;
        }
        case 4:
            for (long long p = first; p < A.n; p += stride) {
                const uint32_t q = start[A.t.cell_of[p]] + A.t.slot[p];
                A.t.tmp_idx[q] = (int)p;
                A.t.tmp_key[q] = order_key(__double_as_longlong(to_f64(z[p])));
            }
            break;
        case 5:  // the cells are claimed one run at a time: after this ticket none is left
            sort_cells<T>(x, y, A.w, nc, g, counts, A.t.tmp_idx, A.t.tmp_key, A.out, counts + nc, s_ent);
            return;
        default:  // a block that began when all was handed out
            return;
        }
    }
}

// Bounding box, on order-preserving integer keys (binary64 compares would hold the
// narrow binary64 pipe).
__device__ __forceinline__ uint32_t order_key32(int b)
{
    return b < 0 ? ~(uint32_t)b : ((uint32_t)b | 0x80000000u);
}
__device__ __forceinline__ unsigned long long key_of(double v) { return order_key(__double_as_longlong(v)); }
__device__ __forceinline__ uint32_t key_of(float v) { return order_key32(__float_as_int(v)); }
__device__ __forceinline__ bool finite_bits(double v)
{
    return (__double_as_longlong(v) & 0x7ff0000000000000ll) != 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool finite_bits(float v)
{
    return (__float_as_int(v) & 0x7f800000) != 0x7f800000;
}
__device__ __forceinline__ unsigned long long wide_key(unsigned long long k) { return k; }
__device__ __forceinline__ unsigned long long wide_key(uint32_t k)
{
    const uint32_t b = (k >> 31) ? (k & 0x7fffffffu) : ~k;
    return key_of(f2d(__uint_as_float(b)));
}

template <class T>
__global__ void k_bbox(const T *__restrict__ x, const T *__restrict__ y, const T *__restrict__ z,
                       long long n, unsigned long long *__restrict__ out /* 6: min xyz, max xyz */,
                       unsigned *__restrict__ err)
{
    using K = decltype(key_of(T(0)));
    K lo[3] = {~K(0), ~K(0), ~K(0)}, hi[3] = {K(0), K(0), K(0)};
    bool bad = false;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        const T v[3] = {x[p], y[p], z[p]};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (!finite_bits(v[a])) {
                bad = true;
                continue;
            }
            const K k = key_of(v[a]);
            lo[a] = min(lo[a], k);
            hi[a] = max(hi[a], k);
        }
    }
    if (bad)
        atomicOr(err, ERR_COORD);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo[a] = min(lo[a], (K)__shfl_xor_sync(FULL, lo[a], o));
            hi[a] = max(hi[a], (K)__shfl_xor_sync(FULL, hi[a], o));
        }
    }
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (lo[a] <= hi[a]) {
                atomicMin(&out[a], wide_key(lo[a]));
                atomicMax(&out[3 + a], wide_key(hi[a]));
            }
    }
}

inline int grid_blocks(long long n, int threads, int sms)
{
    long long b = (n + threads - 1) / threads;
    long long cap = (long long)sms * 16;
    if (b > cap)
        b = cap;
    return (int)(b < 1 ? 1 : b);
}

// ============================================================ batched gridding
// The same stages for every catalogue (segment) of a batch, one launch each:
// a stage's blocks are split among the segments by a prefix array, and the
// counting sort's offsets come from one scan over the segments' concatenated
// padded counts (each segment's ncells + 1 entries, the last one 0), from which
// every segment's cell_start is its slice minus the slice's first value.

// Segment of this block: the largest s with pre[s] <= blockIdx.x (segments
// without blocks of this shape are passed over).  Every thread must call it.
__device__ __forceinline__ int block_seg(const unsigned *pre, int nseg)
{
    __shared__ int s_seg;
    if (threadIdx.x == 0) {
        int lo = 0, hi = nseg - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (pre[mid] <= blockIdx.x)
                lo = mid;
            else
                hi = mid - 1;
        }
        s_seg = lo;
    }
    __syncthreads();
    return s_seg;
}

// Segment holding entry c of the concatenated per-cell arrays.
__device__ __forceinline__ int seg_of_entry(const GridBatch &B, long long c)
{
    int lo = 0, hi = B.nseg - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (B.seg[mid].c0 <= c)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

__global__ void __launch_bounds__(256) kb_assign(const GridBatch B)
{
    __shared__ Geom g;
    const int s = block_seg(B.pre[GB_POINTS], B.nseg);
    const GridSeg &S = B.seg[s];
    static_assert(sizeof(Geom) % 4 == 0, "geometry copied as words");
    for (int q = threadIdx.x; q < (int)(sizeof(Geom) / 4); q += blockDim.x)
        reinterpret_cast<int *>(&g)[q] = reinterpret_cast<const int *>(B.geom + S.job)[q];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const long long p = (long long)(blockIdx.x - B.pre[GB_POINTS][s]) * blockDim.x + threadIdx.x;
    const bool live = p < S.n;
    uint32_t cell = 0xffffffffu;
    if (live) {
        float fx, fy, fz;
        bool ok;
        if (S.f32)
            ok = coord(static_cast<const float *>(S.x)[p], 0, g, fx) &
                 coord(static_cast<const float *>(S.y)[p], 1, g, fy) &
                 coord(static_cast<const float *>(S.z)[p], 2, g, fz);
        else
            ok = coord(static_cast<const double *>(S.x)[p], 0, g, fx) &
                 coord(static_cast<const double *>(S.y)[p], 1, g, fy) &
                 coord(static_cast<const double *>(S.z)[p], 2, g, fz);
        if (!ok) {
            atomicOr(S.err, ERR_COORD);
            fx = fy = fz = 0.0f;
        }
        const int cx = cell_index_f(fx, g.inv_wf[0], g.ncx);
        const int cy = cell_index_f(fy, g.inv_wf[1], g.ncy);
        const int cz = cell_index_f(fz, g.inv_wf[2], g.nz);
        cell = (uint32_t)(((long long)(cx * g.ncy + cy)) * g.nz + cz);
    }
    // one segment per block: equal cells are equal entries
    const unsigned same = __match_any_sync(FULL, cell);
    const int leader = __ffs(same) - 1;
    uint32_t b0 = 0;
    if (live && lane == leader)
        b0 = atomicAdd(&B.counts[S.c0 + cell], (uint32_t)__popc(same));
    b0 = __shfl_sync(FULL, b0, leader);
    if (live) {
        S.cell_of[p] = cell;
        S.slot[p] = b0 + (uint32_t)__popc(same & ((1u << lane) - 1u));
    }
}

// One warp per column: its cells' counts into the concatenated padded counts, the
// padding that rounds the column up to a multiple of COL_PAD in its last cell; the
// last column also zeroes the segment's extra entry.
__global__ void __launch_bounds__(256) kb_colpad(const GridBatch B)
{
    const int s = block_seg(B.pre[GB_COLWARPS], B.nseg);
    const GridSeg &S = B.seg[s];
    const Geom &g = B.geom[S.job];
    const int lane = threadIdx.x & 31, ncols = g.ncols, nz = g.nz;
    const int col = (int)(blockIdx.x - B.pre[GB_COLWARPS][s]) * 8 + (int)(threadIdx.x >> 5);
    if (col >= ncols)
        return;
    const uint32_t *count = B.counts + S.c0;
    uint32_t *padded = B.scan + S.c0;
    const long long c0 = (long long)col * nz;
    uint32_t tot = 0;
    for (int z = lane; z < nz; z += 32) {
        const uint32_t v = count[c0 + z];
        padded[c0 + z] = v;
        tot += v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        tot += __shfl_xor_sync(FULL, tot, o);
    const uint32_t pd = (COL_PAD - (tot & (COL_PAD - 1u))) & (COL_PAD - 1u);
    __syncwarp();
    if (lane == 0) {
        S.pad[col] = pd;
        S.out.colbox[col] = empty_box();
        padded[c0 + nz - 1] += pd;
        if (col == ncols - 1)
            padded[g.ncells] = 0u;
    }
}

// cell_start of every segment: its slice of the scan minus the slice's first value.
__global__ void __launch_bounds__(256) kb_cellstart(const GridBatch B)
{
    const int s = block_seg(B.pre[GB_CELLS], B.nseg);
    const GridSeg &S = B.seg[s];
    const long long k = (long long)(blockIdx.x - B.pre[GB_CELLS][s]) * blockDim.x + threadIdx.x;
    if (k <= B.geom[S.job].ncells)
        S.out.cell_start[k] = B.scan[S.c0 + k] - B.scan[S.c0];
}

__global__ void __launch_bounds__(256) kb_scatter(const GridBatch B)
{
    const int s = block_seg(B.pre[GB_POINTS], B.nseg);
    const GridSeg &S = B.seg[s];
    const long long p = (long long)(blockIdx.x - B.pre[GB_POINTS][s]) * blockDim.x + threadIdx.x;
    if (p >= S.n)
        return;
    const uint32_t q = S.out.cell_start[S.cell_of[p]] + S.slot[p];
    const double zv = S.f32 ? f2d(static_cast<const float *>(S.z)[p]) : static_cast<const double *>(S.z)[p];
    S.tmp_idx[q] = (int)p;
    S.tmp_key[q] = order_key(__double_as_longlong(zv));
}

__device__ __forceinline__ void put_seg(const GridBatch &B, const GridSeg &S, uint32_t d, int iq,
                                        unsigned long long kq, unsigned &wm, ColBox &box)
{
    const Geom &g = B.geom[S.job];
    if (S.f32)
        put_entry(static_cast<const float *>(S.x), static_cast<const float *>(S.y), nullptr, g, d, iq, kq, S.out,
                  wm, box);
    else
        put_entry(static_cast<const double *>(S.x), static_cast<const double *>(S.y), nullptr, g, d, iq, kq,
                  S.out, wm, box);
}

// sort_cells over the concatenated cells of every segment (the cells of a claim may
// belong to different segments; a segment's extra entry has no points).
__global__ void __launch_bounds__(SORT_THREADS) kb_sort_cells(const GridBatch B)
{
    __shared__ ulonglong2 s_ent[SORT_THREADS / 32][SORT_BUF];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned per = claim_cells(B.ctot);
    unsigned wm = 0;
    for (;;) {
        unsigned v = 0u;
        if (lane == 0)
            v = atomicAdd(B.counts + B.ctot, per);  // the next run of entries (zeroed with the counts)
        const long long c = (long long)__shfl_sync(FULL, v, 0) + lane;
        if (c - lane >= B.ctot)
            break;
        int sg = 0, col = -1;
        uint32_t n = 0u, s = 0u;
        if ((unsigned)lane < per && c < B.ctot && (n = B.counts[c]) != 0u) {
            sg = seg_of_entry(B, c);
            const long long cell = c - B.seg[sg].c0;
            s = B.seg[sg].out.cell_start[cell];
            col = B.seg[sg].col0 + (int)cell / B.geom[B.seg[sg].job].nz;
        }
        sort_run(n, s, col, lane, s_ent[wid],
                 [&](int k, int ck) {
                     const GridSeg *S = B.seg + __shfl_sync(FULL, sg, k);
                     return SegSrc{{S->tmp_key, S->tmp_idx, S->out.colbox + (ck - S->col0)}, S};
                 },
                 [&](const SegSrc &src, uint32_t d, int iq, unsigned long long kq, ColBox &box) {
                     put_seg(B, *src.seg, d, iq, kq, wm, box);
                 });
    }
}

__global__ void __launch_bounds__(256) kb_padfill(const GridBatch B)
{
    const int s = block_seg(B.pre[GB_COLWARPS], B.nseg);
    const GridSeg &S = B.seg[s];
    const Geom &g = B.geom[S.job];
    const int col = (int)(blockIdx.x - B.pre[GB_COLWARPS][s]) * 8 + (int)(threadIdx.x >> 5);
    if (col < g.ncols)
        pad_column(S.out, col, S.out.cell_start[(long long)col * g.nz],
                   S.out.cell_start[(long long)(col + 1) * g.nz], S.pad[col], threadIdx.x & 31);
}

template <class T>
cudaError_t build_grid_t(const GridArgs &A, int sms, cudaStream_t st)
{
    int occ = 0;
    const cudaError_t e = occupancy(k_grid<T>, 0, occ);
    if (e)
        return e;
    if (occ < 1)
        return cudaErrorInvalidConfiguration;
    // a thread per point or cell, a warp per column; no more blocks than fit at once
    const long long work = std::max(A.n, std::max(A.g.ncells, 32ll * A.g.ncols));
    const long long blocks = std::min<long long>((long long)sms * occ, (work + SORT_THREADS - 1) / SORT_THREADS);
    k_grid<T><<<(unsigned)std::max(blocks, 1ll), SORT_THREADS, 0, st>>>(A);
    return cudaGetLastError();
}

template <class T>
cudaError_t bbox_t(const void *x, const void *y, const void *z, long long n,
                   unsigned long long *out6, int sms, unsigned *err, cudaStream_t st)
{
    if (n <= 0)
        return cudaSuccess;
    k_bbox<T><<<grid_blocks(n, 256, sms), 256, 0, st>>>((const T *)x, (const T *)y, (const T *)z, n,
                                                         out6, err);
    return cudaGetLastError();
}

}  // namespace

cudaError_t build_grid(cf_dtype dt, const void *x, const void *y, const void *z, const double *w,
                       long long n, const Geom &g, const GridTemps &t, Gridded &out, int sms,
                       unsigned *err, unsigned long long *tickets, uint32_t flags, cudaStream_t st)
{
    out.n = n;
    const GridArgs A{x, y, z, w, n, g, t, out, err, tickets, (flags & CF_FLAG_DEBUG_STALL_GRID) != 0};
    return dt == CF_FLOAT32 ? build_grid_t<float>(A, sms, st) : build_grid_t<double>(A, sms, st);
}

int grid_max_blocks(int sms) { return sms * 8; }  // 2,048 threads per SM

cudaError_t launch_bbox(cf_dtype dt, const void *x, const void *y, const void *z, long long n,
                        unsigned long long *out6, int sms, unsigned *err, cudaStream_t st)
{
    return dt == CF_FLOAT32 ? bbox_t<float>(x, y, z, n, out6, sms, err, st)
                            : bbox_t<double>(x, y, z, n, out6, sms, err, st);
}

long long scan_block_sums(long long n)
{
    return (n + SCAN_ITEMS - 1) / SCAN_ITEMS + 1;  // + the grand total
}

unsigned grid_batch_blocks(int k, long long n, const Geom &g)
{
    switch (k) {
    case GB_POINTS:
        return (unsigned)((n + 255) / 256);
    case GB_COLWARPS:
        return (unsigned)((g.ncols + 7) / 8);
    default:
        return (unsigned)((g.ncells + 1 + 255) / 256);
    }
}

cudaError_t build_grid_batch(const GridBatch &B, int sms, cudaStream_t st)
{
    cudaError_t e;
    if (B.nseg < 1 || B.ctot < 1)
        return cudaSuccess;
    if ((e = cudaMemsetAsync(B.counts, 0, sizeof(uint32_t) * (B.ctot + 1), st)))  // + the sort's claim counter
        return e;
    if (B.blocks[GB_POINTS])
        kb_assign<<<B.blocks[GB_POINTS], 256, 0, st>>>(B);
    kb_colpad<<<B.blocks[GB_COLWARPS], 256, 0, st>>>(B);
    const long long nb = (B.ctot + SCAN_ITEMS - 1) / SCAN_ITEMS;
    k_scan_blocks<<<(unsigned)nb, SCAN_THREADS, 0, st>>>(B.scan, B.scan, B.ctot, B.bsum);
    k_scan_sums<<<1, SCAN_THREADS, 0, st>>>(B.bsum, nb, B.bsum + nb);
    k_scan_add<<<(unsigned)((B.ctot + 255) / 256), 256, 0, st>>>(B.scan, B.ctot, B.bsum);
    kb_cellstart<<<B.blocks[GB_CELLS], 256, 0, st>>>(B);
    if (B.blocks[GB_POINTS]) {
        kb_scatter<<<B.blocks[GB_POINTS], 256, 0, st>>>(B);
        const long long cwarps = std::min<long long>((B.ctot + 1) / 2, (long long)sms * 64);
        kb_sort_cells<<<(unsigned)((cwarps * 32 + SORT_THREADS - 1) / SORT_THREADS), SORT_THREADS, 0, st>>>(B);
    }
    kb_padfill<<<B.blocks[GB_COLWARPS], 256, 0, st>>>(B);
    return cudaGetLastError();
}

double decode_dkey(unsigned long long k)
{
    const unsigned long long b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    double v;
    memcpy(&v, &b, sizeof(v));
    return v;
}

}  // namespace cf
