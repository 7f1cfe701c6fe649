// Batched counting: the chunk tasks (tasks.cuh) of many jobs -- catalogues of
// uneven sizes, bins, modes -- in one persistent launch per kind of count.
//
// A CTA attaches to a job: it loads the job's tables, its warps claim chunks from
// the job's counter until none is left, and the CTA adds its histogram to the
// job's.  Then it moves on to the next job that nobody has begun, or that has
// enough left to be worth loading its tables for.  The jobs are listed from the
// largest down and the CTAs start spread over them in proportion to their
// estimated work, so a large job has many CTAs from the start and a small one is
// done by a single CTA, which loads its tables once.  A CTA leaves a job only when
// all its chunks are claimed, so every job is finished; nobody waits for anybody.
//
// Measured (a run's device time, graph replay, GB300), before -- one kernel for all
// kinds, CTAs claiming column pairs from one queue over all jobs, so that nearly
// every CTA loaded nearly every job's tables -- and now: 480 jobs of 200 to 8,000
// points 6.5 -> 0.97 ms; 48 jobs of 12,500 to 500,000 points 283 -> 43.6 ms (with
// every chunk of a dense job one task the last tasks ran alone for a third of the
// time: 75 ms; all kinds on one stream 49 ms); 100 jobs 140 -> 2.1 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <numeric>
#include <vector>

#include "count32.cuh"
#include "countrp32.cuh"
#include "cull64.cuh"

namespace cf {

namespace {

// CTAs per SM of the binary64 counts beside float32 counts (of three in all).
constexpr int F64_BESIDE = 2;

// Fewest unclaimed tasks for which a CTA joins a job that others work on.
constexpr unsigned JOIN_TASKS = 4 * WARPS;

// Tasks of a job: all chunks are split where a warp gets few of them (plan_batch),
// so that its warps end together; else the last eighth.
__device__ __forceinline__ TaskSplit batch_split(const PairParams &P, unsigned ch)
{
    const unsigned nchunk = P.A.cell_start[P.g.ncells] / ch;
    return TaskSplit(nchunk, (unsigned)P.parts, P.split_all != 0);
}

// Table barrier of a path: the float32 counts load their table through it.
template <class Path>
__device__ __forceinline__ bool batch_load(const PairParams &P, unsigned char *smem,
                                           typename Path::State &st, unsigned &phase)
{
    const bool ok = Path::load(P, smem, st, phase);
    phase ^= 1u;
    return ok;
}

template <class Path, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) k_batch(const PairParams *__restrict__ jobs,
                                                         const int *__restrict__ list,
                                                         const int *__restrict__ start, int n)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_next;
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) {
        mbar_init(reinterpret_cast<uint64_t *>(smem), 1);
        fence_mbar_init();
    }
    __syncthreads();
    unsigned phase = 0u;
    typename Path::State st;
    for (int cur = start[blockIdx.x]; cur >= 0;) {
        const PairParams &P = jobs[list[cur]];
        if (!batch_load<Path>(P, smem, st, phase))
            return;  // the table never came: the job's error word says so
        const TaskSplit split = batch_split(P, Path::CH);
        unsigned nxt = 0;
        if (lane == 0)
            nxt = atomicAdd(P.item_counter, 1u);
        for (unsigned t = __shfl_sync(FULL, nxt, 0); t < split.ntask; t = __shfl_sync(FULL, nxt, 0)) {
            if (lane == 0)
                nxt = atomicAdd(P.item_counter, 1u);
            unsigned c, part, parts;
            split.task(t, c, part, parts);
            Path::task(P, smem, st, c, part, parts);
        }
        Path::fini(P, smem, st);
        __syncthreads();
        if (tid < 32) {  // the next job, 32 looked at together
            int next = -1;
            for (int k0 = 1; k0 < n && next < 0; k0 += 32) {
                const int k = k0 + lane;
                bool take = false;
                if (k < n) {
                    const PairParams &Q = jobs[list[(cur + k) % n]];
                    const unsigned done = *reinterpret_cast<volatile unsigned *>(Q.item_counter);
                    const unsigned all = batch_split(Q, Path::CH).ntask;
                    take = done < all && (done == 0u || all - done >= JOIN_TASKS);
                }
                const unsigned m = __ballot_sync(FULL, take);
                if (m)
                    next = (cur + k0 + __ffs(m) - 1) % n;
            }
            if (lane == 0)
                s_next = next;
        }
        __syncthreads();
        cur = s_next;
        __syncthreads();
    }
}

// The neighbour lists of every job: job j owns blocks [pre[j], pre[j + 1]) of 8
// columns.
__global__ void __launch_bounds__(256) k_neighbours_batch(const PairParams *__restrict__ jobs,
                                                          const unsigned *__restrict__ pre, int njobs)
{
    __shared__ int s_job;
    if (threadIdx.x == 0) {
        int lo = 0, hi = njobs - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (pre[mid] <= blockIdx.x)
                lo = mid;
            else
                hi = mid - 1;
        }
        s_job = lo;
    }
    __syncthreads();
    const int j = s_job;
    neighbours_body(jobs[j], (int)(blockIdx.x - pre[j]) * 8 + (int)(threadIdx.x >> 5), threadIdx.x & 31);
}

// One kernel per group of jobs.
struct Group {
    const void *kern;
    int ch;  // primaries per chunk
};

template <class Path, int MINB>
Group group()
{
    return Group{(const void *)k_batch<Path, MINB>, Path::CH};
}

Group group_of(int path)
{
    switch (path) {
    case BATCH_XI32: return group<Count32<16, 2, false, false, 0>, 3>();
    case BATCH_XI32 + BATCH_LIN: return group<Count32<16, 2, false, false, 1>, 3>();
    case BATCH_XI32_8x2: return group<Count32<8, 2, false, false, 0>, 3>();
    case BATCH_XI32_8x2 + BATCH_LIN: return group<Count32<8, 2, false, false, 1>, 3>();
    case BATCH_XI32_16x1: return group<Count32<16, 1, false, false, 0>, 3>();
    case BATCH_XI32_16x1 + BATCH_LIN: return group<Count32<16, 1, false, false, 1>, 3>();
    case BATCH_XI32_32x1: return group<Count32<32, 1, false, false, 0>, 3>();
    case BATCH_XI32_32x1 + BATCH_LIN: return group<Count32<32, 1, false, false, 1>, 3>();
    case BATCH_RPPI32: return group<CountRp32<16, 2, false, false, 0>, 3>();
    case BATCH_RPPI32 + BATCH_LIN: return group<CountRp32<16, 2, false, false, 1>, 3>();
    case BATCH_XI64: return group<Cull64<0, false, false, 2>, 3>();
    default: return group<Cull64<1, false, false, 2>, 3>();
    }
}

}  // namespace

int batch_path(const PairParams &P, int f64, int chunk, int pp)
{
    if (f64)
        return P.kind == 0 ? BATCH_XI64 : BATCH_RPPI64;
    const int lin = P.lut_lin ? BATCH_LIN : 0;
    if (P.kind == 1)
        return BATCH_RPPI32 + lin;
    if (pp == 2 && chunk == 8)
        return BATCH_XI32_8x2 + lin;
    if (pp == 1 && chunk == 16)
        return BATCH_XI32_16x1 + lin;
    if (pp == 1 && chunk == 32)
        return BATCH_XI32_32x1 + lin;
    return BATCH_XI32 + lin;
}

int batch_smem(PairParams &P, int path)
{
    if (path == BATCH_XI64 || path == BATCH_RPPI64)
        return plan_count64(P);
    return P.kind == 0 ? count32_smem(P.nbins) : countrp32_smem(P.nbins, P.npibins);
}

// Per kind of count its jobs from the largest down and the CTAs' first jobs: CTA b
// of B starts at the job that holds the share (b + 1/2) / B of the group's estimated work
// (weight: the points times the secondaries in reach, and a fixed part per chunk).
// Also every job's task split, for the warps of its share of the CTAs (at least one).
cudaError_t plan_batch(const std::vector<int> &path, const std::vector<int> &smem,
                       const std::vector<double> &work, int sms, std::vector<PairParams> &jobs,
                       BatchPlan &plan)
{
    plan = BatchPlan{};
    std::vector<int> order(path.size());
    std::iota(order.begin(), order.end(), 0);
    std::sort(order.begin(), order.end(), [&](int a, int b) {
        return path[a] != path[b] ? path[a] < path[b] : work[a] != work[b] ? work[a] > work[b] : a < b;
    });
    struct Kind {
        BatchLaunch g;
        int per_sm, f64;
        double total;
    };
    std::vector<Kind> kinds;
    int has[2] = {0, 0};
    for (size_t k = 0; k < order.size();) {
        Kind q{};
        BatchLaunch &g = q.g;
        g.path = path[order[k]];
        g.first = (int)k;
        for (; k < order.size() && path[order[k]] == g.path; ++k) {
            g.smem = std::max(g.smem, smem[order[k]]);
            q.total += work[order[k]];
            ++g.n;
        }
        cudaError_t e = occupancy_of(group_of(g.path).kern, g.smem, q.per_sm);
        if (e)
            return e;
        if (q.per_sm < 1)
            return cudaErrorInvalidConfiguration;
        // both streams' CTAs share SMs: one split of the L1 for all, the largest
        if ((e = cudaFuncSetAttribute(group_of(g.path).kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                      cudaSharedmemCarveoutMaxShared)))
            return e;
        q.f64 = g.path == BATCH_XI64 || g.path == BATCH_RPPI64;
        has[q.f64] = 1;
        for (int j = g.first; j < g.first + g.n; ++j) {
            PairParams &P = jobs[order[j]];
            const double warps = std::max(1.0, work[order[j]] / q.total * sms * q.per_sm) * WARPS;
            const double chunks = (double)(P.A.n + (long long)P.g.ncols * (COL_PAD / 2)) / group_of(g.path).ch + 1.0;
            P.parts = task_parts(chunks, warps, P.nstencil);
            P.split_all = chunks < 8.0 * warps ? 1 : 0;
        }
        kinds.push_back(q);
    }
    const auto add = [&](const Kind &q, int per_sm, int side) {
        if (per_sm < 1)
            return;
        BatchLaunch g = q.g;
        g.blocks = sms * per_sm;
        g.side = side;
        g.start0 = (int)plan.start.size();
        double sum = 0.0;
        int j = -1;
        for (int b = 0; b < g.blocks; ++b) {
            while (j + 1 < g.n && (j < 0 || sum < q.total * (b + 0.5) / g.blocks))
                sum += work[order[g.first + ++j]];
            plan.start.push_back(j);
        }
        plan.launches.push_back(g);
    };
    // Binary64 jobs beside float32 jobs: the binary64 counts wait for their pipe and
    // leave four fifths of the issue slots, the float32 counts issue and leave that pipe
    // idle.  So the binary64 kinds run on a second stream with F64_BESIDE CTAs per SM, the
    // float32 kinds with the rest of theirs; each stream ends with the other's
    // kinds in what room it had, which join the jobs that are not done.  Measured (graph
    // replay, one stream / two with 1 / 2 CTAs per SM): 48 jobs of 12,500 to 500,000 points
    // 49.3 / 47.8 / 44.7 ms; 480 small jobs 1.042 / 0.979 / 0.967; 900 tiny jobs 0.613 / 0.496 /
    // 0.527; 100 jobs 2.18 / 2.04 / 2.09.
    plan.forked = has[0] && has[1];
    if (!plan.forked) {
        for (const Kind &q : kinds)
            add(q, q.per_sm, 0);
    } else {
        for (int pass = 0; pass < 2; ++pass)  // its own kinds first, then the other's
            for (int side = 1; side >= 0; --side)
                for (const Kind &q : kinds) {
                    if (q.f64 != (pass ? !side : side))
                        continue;
                    const int beside = std::min(F64_BESIDE, std::max(1, q.per_sm - 1));
                    add(q, side ? beside : std::max(pass ? 0 : 1, q.per_sm - beside), side);
                }
    }
    plan.list = order;
    return cudaSuccess;
}

cudaError_t launch_neighbours_batch(const PairParams *jobs, const unsigned *pre, int njobs, unsigned blocks,
                                    cudaStream_t st)
{
    if (blocks == 0 || njobs < 1)
        return cudaSuccess;
    k_neighbours_batch<<<blocks, 256, 0, st>>>(jobs, pre, njobs);
    return cudaGetLastError();
}

cudaError_t launch_batch(const BatchPlan &plan, const PairParams *jobs, const int *list, const int *start,
                         const BatchSide &side, cudaStream_t st)
{
    cudaError_t e = cudaSuccess;
    if (plan.forked && ((e = cudaEventRecord(side.fork, st)) || (e = cudaStreamWaitEvent(side.stream, side.fork, 0))))
        return e;
    for (size_t k = 0; k < plan.launches.size() && !e; ++k) {
        const BatchLaunch &g = plan.launches[k];
        const int *l = list + g.first, *s = start + g.start0;
        int n = g.n;
        void *args[] = {(void *)&jobs, (void *)&l, (void *)&s, (void *)&n};
        e = cudaLaunchKernel(group_of(g.path).kern, dim3(g.blocks), dim3(THREADS), args, (size_t)g.smem,
                             g.side ? side.stream : st);
    }
    if (plan.forked) {  // the streams join also after a failed launch
        const cudaError_t r = cudaEventRecord(side.join, side.stream), w = cudaStreamWaitEvent(st, side.join, 0);
        e = e ? e : r ? r : w;
    }
    return e;
}

}  // namespace cf
