// Host interface of the pair kernels (pairs.cu).
#pragma once

#include <vector>

#include "cf_internal.cuh"

namespace cf {

__host__ __device__ inline int align_up(int v, int a) { return (v + a - 1) / a * a; }

constexpr int SMEM_MAX = 232448;  // dynamic shared memory a CTA may opt in to (227 KB)

struct PairLaunch {
    int f64;      // 1: binary64 counts
    int chunk;    // primary lanes per warp chunk (8, 16 or 32)
    int pp;       // primaries per lane (1, 2 or 4; float32 counts)
    int evals;    // count evaluations
    int verify;   // verify float32 decisions against binary64
    int blocks;   // persistent CTAs
    int smem;     // dynamic shared memory bytes
    int kernels;  // kernels the launch issued (neighbour lists, pair kernel)
};

// Chunk tasks (tasks.cuh): the neighbour lists of d1's columns (P.nbr,
// P.nbr_count; kept pairs added to *P.work_count), and the float32 DD(r) counts.
cudaError_t launch_neighbours(const PairParams &P, cudaStream_t st);
cudaError_t launch_count32(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st);
int count32_smem(int nbins);
// The same with one histogram word for two pairs, where that is faster.
bool count32_paired(const PairParams &P, const PairLaunch &L);
cudaError_t launch_count32_paired(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st);
// Float32 DD(rp, pi) counts.
cudaError_t launch_countrp32(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st);
int countrp32_smem(int nbins, int npibins);
// Binary64 counts: offsets and histogram copies into P, bytes of shared memory back.
int plan_count64(PairParams &P);
cudaError_t launch_count64(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st);

// Float32 sums: DD(r), DD(rp, pi).
cudaError_t launch_sums32(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st);
cudaError_t launch_sumsrp32(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st);

// The kernels of one count: neighbour lists, then the pair kernel of its kind.
cudaError_t launch_pairs(const PairParams &P, PairLaunch &L, int sms, cudaStream_t st);

// ---- batched launch: one persistent kernel per kind of count
enum : int {
    BATCH_XI32 = 0,       // float32 DD(r), chunks of 16 lanes x 2 primaries
    BATCH_XI64 = 1,
    BATCH_RPPI32 = 2,
    BATCH_RPPI64 = 3,
    BATCH_XI32_8x2 = 4,   // float32 DD(r) with the other tuned shapes
    BATCH_XI32_16x1 = 5,
    BATCH_XI32_32x1 = 6,
    BATCH_LIN = 8,        // added: table cells linear in the squared distance
};
constexpr int BATCH_MAX = 1024;  // jobs per batched launch

// A launch over the jobs of one kind of count: list[first .. first + n), CTA b's first
// job (index into that range) at start[start0 + b]; side: on the second stream.
struct BatchLaunch {
    int path, first, n, blocks, start0, smem, side;
};
struct BatchPlan {
    std::vector<BatchLaunch> launches;  // in the order they are issued
    bool forked;                        // some are on the second stream
    std::vector<int> list, start;
};

// The second stream of a plan that forks and the events that bracket it.
struct BatchSide {
    cudaStream_t stream;
    cudaEvent_t fork, join;
};

// Path of a job: float32 (float32 DD(r) in the kernel shape chunk x pp: 16 x 2,
// 8 x 2, 16 x 1 or 32 x 1, else 16 x 2) or binary64, DD(r) or DD(rp, pi);
// unweighted only.  Needs P's table (lut_lin).
int batch_path(const PairParams &P, int f64, int chunk = 16, int pp = 2);

// Shared memory of a job on that path; its offsets into P.
int batch_smem(PairParams &P, int path);

// Groups, lists and first jobs from every job's path, shared memory and estimated
// work; the jobs' task splits into their parameters.
cudaError_t plan_batch(const std::vector<int> &path, const std::vector<int> &smem,
                       const std::vector<double> &work, int sms, std::vector<PairParams> &jobs,
                       BatchPlan &plan);

// The neighbour lists of njobs jobs (device parameter array) in one launch; job j
// owns blocks [pre[j], pre[j + 1]) of 8 columns, blocks = pre[njobs].
cudaError_t launch_neighbours_batch(const PairParams *jobs, const unsigned *pre, int njobs, unsigned blocks,
                                    cudaStream_t st);

// The kernels of a plan; list and start are device copies of the plan's.
cudaError_t launch_batch(const BatchPlan &plan, const PairParams *jobs, const int *list, const int *start,
                         const BatchSide &side, cudaStream_t st);

}  // namespace cf
