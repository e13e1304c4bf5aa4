// Combine step: average state, row norms of the averaged sketch, median, H, trigger
// (Algorithm 1: the state average and the variance test; Theorem 1 for SketchFDA, Theorem 2 for LinearFDA).
//
// Bound: latency.  The K x (2 + l*m) floats are a few kilobytes to a megabyte; what takes time is
// the chain launch - loads - reductions - (meeting of the blocks) - median - result.  So a thread
// asks for eight workers' values of a column before it adds any, and a warp meets the others once.
// Tables that a block reads in up to kOneBlockTrips round trips are taken by one block (a ticket and a second
// trip to L2 cost more than that); larger ones by one block per 64 columns of a row, its threads
// splitting the workers four ways, and the block that finishes last (a ticket counter, no waiting)
// takes the median.  The median comes from the ranks of the row norms, all rows at once.
// fp64 accumulation in a fixed order, so the result is reproducible.
#include "fda_internal.h"

namespace {

constexpr int kThreads = 1024;             // of the block that takes everything
constexpr int kUnitColumns = 64;           // columns of a block that takes a part of a row,
constexpr int kUnitSlices = 4;             // and the slices of workers its threads split into
constexpr int kUnitThreads = kUnitColumns * kUnitSlices;
// Round trips (batches of eight workers of a warp's 32 columns, one after the other) that cost one block what a
// meeting of several costs.  Measured, one block and several, back to back: two trips 3.54 and 3.79 us (16 x 64, K = 8),
// 3.80 and 3.72 (5 x 250, K = 8); three 3.70 and 3.95 (3 x 100, K = 20); four 4.45 and 3.73 (5 x 250, K = 10), 4.46 and
// 3.73 (7 x 500, K = 1), 4.25 and 4.08 (3 x 100, K = 27); eleven 7.30 and 4.48 us (8 x 1000, K = 1).  Behind a sketch
// pass the difference at four trips is lost in the chain (a round with 5 x 250, K = 10, d = 1.2M: 49.8 us with either).
constexpr int kOneBlockTrips = 3;
// Partials of a row that the block which takes the median asks for at once, together with the scalars.  Back to back, one after
// the other and all at once: 5 x 250, K = 14 3.71 and 3.56 us, 7 x 500, K = 20 3.99 and 3.84, 8 x 1000, K = 33 5.00 and 4.83, 3 x 100, K = 30
// 4.14 and 3.87.  Through shared memory, a thread each: 4.2, 4.3, 4.4, 3.5; the scalars by a block of their own 3.81, 4.07, 4.61, 3.49.
constexpr int kMeetingBatch = 16;
constexpr int kBatch = 8;                  // workers whose values of a column are asked for at once

struct CombineParams {
    const float *states;
    int K, l, m, chunks;                   // chunks: blocks per sketch row (several blocks only)
    int variant;
    float theta;
    double *scratch;                       // [0..1] S-bar[0..1], then one partial per block
    unsigned int *ticket;                  // 0 between launches
    double inv_k, inv_eps;                 // 1 / K, 1 / (1 + epsilon)
    fda_estimate *est;
    unsigned long long *host;              // mapped host memory (fda_host_estimate) or null,
    unsigned int seq;                      // and the number of this estimate
};

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// sum over the workers first, first + step, ... of one column: eight loads in flight, the eight added
// as a tree (a chain of fp64 additions as long as the loads themselves would follow them), the trees in order
__device__ __forceinline__ double column_sum(const float *col, int first, int step, int K, size_t slen)
{
    double acc = 0.0;
    for (int k = first; k < K; k += kBatch * step) {
        float v[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) v[u] = k + u * step < K ? __ldcg(col + (size_t)(k + u * step) * slen) : 0.f;
        acc += (((double)v[0] + (double)v[1]) + ((double)v[2] + (double)v[3])) +
               (((double)v[4] + (double)v[5]) + ((double)v[6] + (double)v[7]));
    }
    return acc;
}

// sum over the workers of entry e (0, 1): lanes stride the workers, fixed shuffle tree
__device__ __forceinline__ double scalar_sum(const float *states, int K, size_t slen, int e, int lane)
{
    double acc = 0.0;
    for (int k = lane; k < K; k += 32) acc += (double)__ldcg(states + (size_t)k * slen + e);
    return warp_sum(acc);
}

// One warp: lane r < l holds ||row r of the averaged sketch||^2; writes the estimate.
__device__ __forceinline__ void finish(const CombineParams &p, double row, double head0, double head1, int lane)
{
    double est_sq = head1 * head1;
    if (p.variant == FDA_VARIANT_SKETCH) {
        int rank = 0;                      // of this lane's row, ties by row number; NaN behind all numbers, so that
        const bool nan = row != row;       // the ranks are 0 .. l - 1 whatever the rows hold
        for (int q = 0; q < p.l; ++q) {
            const double o = __shfl_sync(0xffffffffu, row, q);
            const bool tie = o == row || (nan && o != o);
            rank += (tie ? q < lane : (o < row || nan)) ? 1 : 0;
        }
        const unsigned lo = __ballot_sync(0xffffffffu, lane < p.l && rank == (p.l - 1) / 2);
        const unsigned hi = __ballot_sync(0xffffffffu, lane < p.l && rank == p.l / 2);
        const double a = __shfl_sync(0xffffffffu, row, lo ? __ffs(lo) - 1 : 0);
        const double b = __shfl_sync(0xffffffffu, row, hi ? __ffs(hi) - 1 : 0);
        est_sq = ((p.l & 1) ? a : 0.5 * (a + b)) * p.inv_eps;
    }
    const double H = head0 - est_sq;
    const int trigger = (H > (double)p.theta) ? 1 : 0;    // decided in fp64, strict '>'
    fda_estimate *est = p.est;
    if (lane == 0) {
        est->mean_sq_norm = (float)head0;
        est->est_sq_norm_of_mean = (float)est_sq;
        est->H = (float)H;
        est->theta = p.theta;
        est->trigger = trigger;
        est->l = p.l;
    }
    const float norm = lane < p.l ? (float)row : 0.f;
    if (lane < FDA_MAX_ROWS) est->row_sq_norm[lane] = norm;
    if (p.host) {      // lane 4 + r: row r; every word carries the estimate's number, so nothing orders the words
        // among each other.  The fence puts *est (and the ticket) in front of them: the host that has read
        // the words may launch a reader of *est on any stream.  It is of system scope, because the observer is the
        // host, and behind the warp's meeting, so that each lane's word follows what all lanes have written.
        // A step at LeNet-5 size takes 23.8 us with it, 22.7 with a fence of device scope, which orders the
        // writes for observers on the GPU only; fence.acq_rel.sys in its place: 23.9 us.
        __syncwarp();
        __threadfence_system();
        const float shifted = __shfl_up_sync(0xffffffffu, norm, 4);
        const uint32_t word = lane == 0 ? __float_as_uint((float)head0) : lane == 1 ? __float_as_uint((float)est_sq)
                            : lane == 2 ? __float_as_uint((float)H) : lane == 3 ? (uint32_t)trigger : __float_as_uint(shifted);
        if (lane < 4 + p.l)
            *reinterpret_cast<volatile unsigned long long *>(p.host + lane) = ((unsigned long long)p.seq << 32) | word;
    }
}

// One block: warp w takes the columns stripe*32 + lane, + 32*stripes, ... of row w % l.
__global__ void __launch_bounds__(kThreads, 1) k_combine_small(const CombineParams p)
{
    __shared__ double part_s[32], head_s[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t slen = 2 + (size_t)p.l * (size_t)p.m;
    const int stripes = p.l > 0 ? 30 / p.l : 0;            // warps per row; the last two warps take the scalars
    fda_grid_wait();
    double part = 0.0;
    if (warp >= 30) {
        const double h = scalar_sum(p.states, p.K, slen, warp - 30, lane) * p.inv_k;
        if (lane == 0) head_s[warp - 30] = h;
    } else if (warp < stripes * p.l) {
        const int i = warp % p.l;
        for (int c = (warp / p.l) * 32 + lane; c < p.m; c += stripes * 32) {
            const double t = column_sum(p.states + 2 + (size_t)i * p.m + c, 0, 1, p.K, slen) * p.inv_k;
            part += t * t;
        }
        part = warp_sum(part);
    }
    if (lane == 0) part_s[warp] = part;
    __syncthreads();
    if (warp != 0) return;
    double row = 0.0;
    if (lane < p.l)
        for (int q = 0; q < stripes; ++q) row += part_s[q * p.l + lane];
    finish(p, row, head_s[0], head_s[1], lane);
}

// Block b: the 64 columns b % chunks of row b / chunks; two warps of block 0 also take the scalars.
__global__ void __launch_bounds__(kUnitThreads) k_combine(const CombineParams p)
{
    __shared__ double slice_s[kUnitThreads], part_s[kUnitColumns / 32];
    __shared__ bool last_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const size_t slen = 2 + (size_t)p.l * (size_t)p.m;
    fda_grid_wait();
    const int i = (int)blockIdx.x / p.chunks, sl = tid / kUnitColumns;
    const int c = ((int)blockIdx.x % p.chunks) * kUnitColumns + tid % kUnitColumns;
    slice_s[tid] = c < p.m ? column_sum(p.states + 2 + (size_t)i * p.m + c, sl, kUnitSlices, p.K, slen) : 0.0;
    if (blockIdx.x == 0 && warp < 2) {
        const double h = scalar_sum(p.states, p.K, slen, warp, lane) * p.inv_k;
        if (lane == 0) { p.scratch[warp] = h; __threadfence(); }
    }
    __syncthreads();
    if (tid < kUnitColumns) {
        double t = 0.0;
#pragma unroll
        for (int q = 0; q < kUnitSlices; ++q) t += slice_s[q * kUnitColumns + tid];
        t *= p.inv_k;
        t = warp_sum(t * t);
        if (lane == 0) part_s[warp] = t;
    }
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
#pragma unroll
        for (int q = 0; q < kUnitColumns / 32; ++q) t += part_s[q];
        p.scratch[2 + blockIdx.x] = t;
        __threadfence();
        last_s = atomicAdd(p.ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last_s || warp != 0) return;
    __threadfence();
    const double head0 = __ldcg(p.scratch), head1 = __ldcg(p.scratch + 1);
    double row = 0.0;
    for (int q0 = 0; q0 < p.chunks; q0 += kMeetingBatch) {
        double v[kMeetingBatch];
#pragma unroll
        for (int q = 0; q < kMeetingBatch; ++q)
            v[q] = lane < p.l && q0 + q < p.chunks ? __ldcg(p.scratch + 2 + lane * p.chunks + q0 + q) : 0.0;
#pragma unroll
        for (int q = 0; q < kMeetingBatch; ++q) row += v[q];
    }
    if (lane == 0) *p.ticket = 0u;                         // ready for the next launch on this context
    finish(p, row, head0, head1, lane);
}

}  // namespace

cudaError_t fda_launch_combine(const fda_ctx *ctx, const float *states, int K, int variant,
                               float epsilon, float theta, fda_estimate *est_dev, unsigned long long *host,
                               unsigned int seq, cudaStream_t s)
{
    CombineParams p{};
    p.states = states; p.K = K; p.l = ctx->l; p.m = ctx->m;
    p.variant = variant; p.theta = theta;
    p.inv_k = 1.0 / (double)K; p.inv_eps = 1.0 / (1.0 + (double)epsilon);
    p.scratch = ctx->combine_scratch; p.ticket = ctx->combine_ticket;
    p.est = est_dev; p.host = host; p.seq = seq;
    // k_combine_small: 30 / l warps to a row, 32 columns a warp
    const int64_t columns = ctx->l > 0 ? 30 / ctx->l * 32 : 1, trips = (ctx->m + columns - 1) / columns * ((K + kBatch - 1) / kBatch);
    if (ctx->l == 0 || trips <= kOneBlockTrips)
        return fda_launch_dependent(k_combine_small, 1, kThreads, 0, s, p);
    p.chunks = (ctx->m + kUnitColumns - 1) / kUnitColumns;
    return fda_launch_dependent(k_combine, ctx->l * p.chunks, kUnitThreads, 0, s, p);
}

// doubles of the context's combine scratch: the two scalars and one partial per block
size_t fda_combine_scratch_doubles(int l, int m) { return 2 + (size_t)l * ((size_t)(m + kUnitColumns - 1) / kUnitColumns); }
