// K-way model average (Section 3: the workers synchronise with an AllReduce of their models,
// the synchronisation step of Algorithm 1): w-bar = (1/K) sum_k w^(k), written to w_t0 and, when broadcasting, to every row.
// Bandwidth-bound streaming kernel; the whole launch is predicated on the trigger word of
// the device-side estimate so that no host round trip is needed between the two calls.
#include "fda_internal.h"
#include "fda_quads.cuh"

namespace {

constexpr int kBatch = 8;   // rows loaded before they are summed (loads in flight per thread)
constexpr int kShiftedBatch = 4;   // the same for rows at any alignment (two loads each)

// block partial of ||delta||^2, fixed order
__device__ __forceinline__ void block_partial(double dsq, double *part)
{
    __shared__ double red[8];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dsq += __shfl_xor_sync(0xffffffffu, dsq, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = dsq;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int wv = 0; wv < 8; ++wv) t += red[wv];
        part[blockIdx.x] = t;
    }
}

// Chunks of a vector in the order in which blocks come free.  With a fixed stride some SMs run ahead of others,
// so that the launch reads and writes rows all over a wide window and ends with few SMs at work; with tickets
// the blocks stay side by side.  A block asks for its next chunk before it works on the one it has.
// ticket[0]: chunks handed out beyond the first of every block, ticket[1]: blocks that are done; both 0 between launches.
template <bool TICKETS>
struct ChunkOrder {
    unsigned int *ticket;
    unsigned int *taken;        // two words of shared memory
    unsigned int c = blockIdx.x;
    int phase = 0;
    __device__ __forceinline__ void ask()
    {
        if (TICKETS && threadIdx.x == 0) taken[phase] = gridDim.x + atomicAdd(ticket, 1u);
    }
    __device__ __forceinline__ void next()
    {
        if (!TICKETS) { c += gridDim.x; return; }
        __syncthreads();
        c = taken[phase];
        phase ^= 1;
    }
    __device__ __forceinline__ void done()
    {
        if (!TICKETS || threadIdx.x != 0) return;
        __threadfence();
        if (atomicAdd(ticket + 1, 1u) == gridDim.x - 1) { ticket[0] = 0u; ticket[1] = 0u; }
    }
};

// XI: also write the unnormalised direction of the global step, delta = w-bar_new - w_t0_old, to
// xi_out and the block's partial of ||delta||^2 to part (Section 3.2: xi is the normalised
// difference of the models of the last two synchronisations).
// TICKETS: chunks by ticket (not with XI: the partials of ||delta||^2 keep a fixed order).
template <bool XI, bool TICKETS>
__global__ void __launch_bounds__(256)
k_average(float *w, int64_t row_stride, int K, int64_t d, float *__restrict__ w_t0,
          const fda_estimate *est, int broadcast, float *__restrict__ xi_out, double *__restrict__ part, unsigned int *ticket)
{
    __shared__ unsigned int taken[2];
    fda_grid_wait();
    if (est != nullptr && est->trigger == 0) return;
    double dsq = 0.0;
    const float inv_k = 1.0f / (float)K;
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nq = d / 4;
    const unsigned int chunks = (unsigned int)((nq + 255) / 256);
    ChunkOrder<TICKETS> order{ticket, taken};
    while (order.c < chunks) {
        order.ask();
        const int64_t q = (int64_t)order.c * 256 + threadIdx.x;
        if (q < nq) {
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int k0 = 0; k0 < K; k0 += kBatch) {
                float4 v[kBatch];
#pragma unroll
                for (int b = 0; b < kBatch; ++b)
                    if (k0 + b < K)
                        v[b] = __ldcs(reinterpret_cast<const float4 *>(w + (size_t)(k0 + b) * row_stride + q * 4));
#pragma unroll
                for (int b = 0; b < kBatch; ++b)
                    if (k0 + b < K) { acc.x += v[b].x; acc.y += v[b].y; acc.z += v[b].z; acc.w += v[b].w; }
            }
            acc.x *= inv_k; acc.y *= inv_k; acc.z *= inv_k; acc.w *= inv_k;
            if (XI) {
                const float4 old = *reinterpret_cast<const float4 *>(w_t0 + q * 4);
                const float4 dl = make_float4(acc.x - old.x, acc.y - old.y, acc.z - old.z, acc.w - old.w);
                *reinterpret_cast<float4 *>(xi_out + q * 4) = dl;
                dsq += (double)(dl.x * dl.x + dl.y * dl.y + dl.z * dl.z + dl.w * dl.w);
            }
            __stcs(reinterpret_cast<float4 *>(w_t0 + q * 4), acc);
            if (broadcast)
                for (int k = 0; k < K; ++k)
                    __stcs(reinterpret_cast<float4 *>(w + (size_t)k * row_stride + q * 4), acc);
        }
        order.next();
    }
    order.done();
    // the d % 4 tail
    for (int64_t j = nq * 4 + t0; j < d; j += nthreads) {
        float acc = 0.f;
        for (int k = 0; k < K; ++k) acc += w[(size_t)k * row_stride + j];
        acc *= inv_k;
        if (XI) {
            const float dl = acc - w_t0[j];
            xi_out[j] = dl;
            dsq += (double)(dl * dl);
        }
        w_t0[j] = acc;
        if (broadcast)
            for (int k = 0; k < K; ++k) w[(size_t)k * row_stride + j] = acc;
    }
    if (XI) block_partial(dsq, part);
}

// The same for rows, w_t0 or xi_out that are not all 16-byte aligned (fda_quads.cuh): a warp takes 32
// consecutive quads in the frame of w_t0; what lies in front of the second quad and behind the
// last but one is left to single floats, one thread each.
// Measured on B200 with broadcast, K = 30, d = 6,964,106 at a pitch of d: 293 us (297 with aligned rows); with
// 32-bit accesses throughout, as before, 346 us; eight rows a batch 310 us.
template <bool XI, bool TICKETS>
__global__ void __launch_bounds__(256)
k_average_shifted(float *w, int64_t row_stride, int K, int64_t d, float *w_t0,
                  const fda_estimate *est, int broadcast, float *__restrict__ xi_out, double *__restrict__ part, unsigned int *ticket)
{
    using namespace fda_quads;
    __shared__ unsigned int taken[2];
    fda_grid_wait();
    if (est != nullptr && est->trigger == 0) return;
    double dsq = 0.0;
    const float inv_k = 1.0f / (float)K;
    const int lane = threadIdx.x & 31;
    const int c0 = first_aligned(w_t0);
    // whole quads 1 .. Q - 1: the windows of all rows around them lie inside [0, d)
    const int64_t Q = d >= c0 + 12 ? (d - c0 - 8) / 4 + 1 : 1;
    const unsigned int chunks = (unsigned int)((Q - 1 + 255) / 256);
    const bool xi_al = XI && misaligned(xi_out + c0) == 0;
    ChunkOrder<TICKETS> order{ticket, taken};
    while (order.c < chunks) {
        order.ask();
        const int64_t q0 = 1 + 32 * ((int64_t)order.c * 8 + (threadIdx.x >> 5));
        if (q0 < Q) {
            const int64_t q = q0 + lane;
            const bool on = q < Q;
            const int64_t j = c0 + 4 * (on ? q : q0);          // lanes past the end repeat the first quad
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int k0 = 0; k0 < K; k0 += kShiftedBatch) {
                Window v[kShiftedBatch];
#pragma unroll
                for (int b = 0; b < kShiftedBatch; ++b)
                    if (k0 + b < K) v[b] = load_window(w + (size_t)(k0 + b) * row_stride + j);
#pragma unroll
                for (int b = 0; b < kShiftedBatch; ++b)
                    if (k0 + b < K) {
                        const float4 x = value(v[b], w + (size_t)(k0 + b) * row_stride + j);
                        acc.x += x.x; acc.y += x.y; acc.z += x.z; acc.w += x.w;
                    }
            }
            acc.x *= inv_k; acc.y *= inv_k; acc.z *= inv_k; acc.w *= inv_k;
            if (XI && on) {
                const float4 old = *reinterpret_cast<const float4 *>(w_t0 + j);
                const float4 dl = make_float4(acc.x - old.x, acc.y - old.y, acc.z - old.z, acc.w - old.w);
                if (xi_al) *reinterpret_cast<float4 *>(xi_out + j) = dl;
                else { xi_out[j] = dl.x; xi_out[j + 1] = dl.y; xi_out[j + 2] = dl.z; xi_out[j + 3] = dl.w; }
                dsq += (double)(dl.x * dl.x + dl.y * dl.y + dl.z * dl.z + dl.w * dl.w);
            }
            if (on) __stcs(reinterpret_cast<float4 *>(w_t0 + j), acc);
            if (broadcast) {
                float4 nx;
                nx.x = __shfl_down_sync(0xffffffffu, acc.x, 1);
                nx.y = __shfl_down_sync(0xffffffffu, acc.y, 1);
                nx.z = __shfl_down_sync(0xffffffffu, acc.z, 1);
                nx.w = 0.f;
                if (on)
                    for (int k = 0; k < K; ++k)
                        store_shifted(w + (size_t)k * row_stride + j, acc, nx, lane == 0, lane == 31 || q + 1 == Q);
            }
        }
        order.next();
    }
    order.done();
    // the ends
    const int64_t head = d < c0 + 4 ? d : c0 + 4, tail = c0 + 4 * Q, n_ends = head + (tail < d ? d - tail : 0);
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n_ends; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = t < head ? t : tail + (t - head);
        float acc = 0.f;
        for (int k = 0; k < K; ++k) acc += w[(size_t)k * row_stride + j];
        acc *= inv_k;
        if (XI) {
            const float dl = acc - w_t0[j];
            xi_out[j] = dl;
            dsq += (double)(dl * dl);
        }
        w_t0[j] = acc;
        if (broadcast)
            for (int k = 0; k < K; ++k) w[(size_t)k * row_stride + j] = acc;
    }
    if (XI) block_partial(dsq, part);
}

// Short vectors: one index per thread, whatever the alignment.  A quad per thread would leave most of
// the SMs' warps without work, and what a thread waits for is a chain of round trips, one per
// batch of rows, so a batch is sixteen rows deep.
template <bool XI>
__global__ void __launch_bounds__(256)
k_average_short(float *w, int64_t row_stride, int K, int64_t d, float *w_t0,
                const fda_estimate *est, int broadcast, float *__restrict__ xi_out, double *__restrict__ part)
{
    constexpr int kDeep = 16;
    fda_grid_wait();
    if (est != nullptr && est->trigger == 0) return;
    double dsq = 0.0;
    const float inv_k = 1.0f / (float)K;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < d; j += (int64_t)gridDim.x * blockDim.x) {
        float acc = 0.f;
        for (int k0 = 0; k0 < K; k0 += kDeep) {
            float v[kDeep];
#pragma unroll
            for (int b = 0; b < kDeep; ++b)
                if (k0 + b < K) v[b] = __ldcs(w + (size_t)(k0 + b) * row_stride + j);
#pragma unroll
            for (int b = 0; b < kDeep; ++b)
                if (k0 + b < K) acc += v[b];
        }
        acc *= inv_k;
        if (XI) {
            const float dl = acc - w_t0[j];
            xi_out[j] = dl;
            dsq += (double)(dl * dl);
        }
        w_t0[j] = acc;
        if (broadcast) {
#pragma unroll 8
            for (int k = 0; k < K; ++k) __stcs(w + (size_t)k * row_stride + j, acc);
        }
    }
    if (XI) block_partial(dsq, part);
}

// xi_out *= 1 / ||delta||  (0 when the step is zero); gated like the average itself
__global__ void __launch_bounds__(256)
k_scale_xi(float *xi_out, int64_t d, const double *part, int nparts,
           const fda_estimate *est)
{
    fda_grid_wait();
    if (est != nullptr && est->trigger == 0) return;
    // the sum of the partials, the same in every block: threads stride them, then a fixed tree
    __shared__ double red[8];
    __shared__ float scale_s;
    double t = 0.0;
    for (int b = threadIdx.x; b < nparts; b += 256) t += __ldcg(part + b);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double sum = 0.0;
        for (int wv = 0; wv < 8; ++wv) sum += red[wv];
        scale_s = sum > 0.0 ? (float)(1.0 / sqrt(sum)) : 0.f;
    }
    __syncthreads();
    const float scale = scale_s;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < d; j += (int64_t)gridDim.x * blockDim.x)
        xi_out[j] *= scale;
}

}  // namespace

cudaError_t fda_launch_average(const fda_ctx *ctx, float *w, int64_t row_stride, int K, int64_t d,
                               float *w_t0, float *xi_out, const fda_estimate *est_dev, uint32_t flags,
                               cudaStream_t s)
{
    const bool vec = ((((uintptr_t)w | (uintptr_t)w_t0 | (uintptr_t)xi_out) & 15u) == 0) && (row_stride % 4 == 0);
    const fda_estimate *gate = (flags & FDA_AVG_UNCONDITIONAL) ? nullptr : est_dev;
    const int broadcast = (flags & FDA_AVG_BROADCAST) ? 1 : 0;
    const int threads = 256;
    // One index per thread on short vectors, up to a number of indices per SM that depends on what the quads cost
    // there: rows at any alignment pay for windows and shifted stores, many rows for the chain of their batches.  Quads of
    // one wave (four blocks to an SM, 4096 indices) catch up; a second wave that is less than half full costs as much as a full
    // one, so behind 4096 indices per SM rows at any alignment go one index per thread once more.  Sixteen rows deep: with 24 or
    // 32 registers keep too few threads on an SM (K = 30, d = 700K 31.8 us, 40 with either).
    // Measured, calls back to back, one index per thread and quads, d in thousands.
    // Aligned, broadcast: K = 12, d = 180 4.3 and 4.5 us; K = 16, 180 5.6 and 6.1; K = 30, 120 6.8 and 10.2, 180 10.2 and 12.6, 260 12.8
    // and 13.5; K = 20, 180 8.3 and 8.4, 260 10.3 and 9.1; K = 60, 180 18.6 and 22.4, 260 23.9 and 24.9, 380 33.4 and 32.9; K = 8, 260 4.5 and 3.8.
    // Without: K = 16, 180 4.0 and 4.1; K = 20, 180 5.7 and 5.0; K = 44, 180 8.3 and 9.4.
    // Any alignment, broadcast: K = 4, 120 3.8 and 3.7, 380 5.4 and 5.3, 520 6.2 and 4.4; K = 6, 260 4.2 and 4.9, 380 5.5 and 5.3; K = 8, 380 6.1 and
    // 6.6, 520 8.5 and 8.2; K = 12, 380 8.3 and 9.4, 520 10.6 and 11.1, 600 11.9 and 11.7; K = 20, 380 14.0 and 14.1, 520 18.3 and 17.6;
    // K = 30, 260 13.1 and 17.3, 520 24.1 and 26.2, 600 27.1 and 27.9; in the second wave K = 8, 700 11.1 and 11.9; K = 10, 700 12.6 and 14.9, 900
    // 15.4 and 16.6; K = 20, 700 23.9 and 26.5, 900 29.8 both; K = 30, 620 28.3 and 37.7, 900 40.5 and 44.5, 1100 50.5 both; K = 60, 700
    // 63.4 and 78, 900 80.7 and 91, 1100 102 and 99.
    // Without: K = 8, 200 3.6 and 3.8, 260 3.8 and 3.7; K = 10, 380 5.4 both; K = 20, 260 7.0 and 7.2, 380 8.8 and 8.1; K = 30, 380 9.7 and 11.4;
    // K = 36, 380 12.7 both, 520 16.5 and 14.5; second wave K = 10, 700 8.2 and 8.5, 900 9.8 and 9.2; K = 20, 620 13.1 both, 700 14.2 and 13.7;
    // K = 44, 700 23.1 and 28.2, 900 28.1 and 30.9.  With xi_out the lines are older ones.
    // (17 to 20 workers: a second batch of up to four rows is a round trip for little, so their lines lie lower: K = 20, 450 15.9 and 14.8)
    const bool many = K >= 10 && !xi_out, rest = K > 16 && K <= 20;
    int64_t per_sm = vec ? (K > 32 ? 1536 : many && broadcast ? 1300 : 768) : K < 8 ? 768 : 1536;
    if (!vec && xi_out && K > 32) per_sm = 4096;
    else if (!vec && many) per_sm = broadcast ? (rest ? 2600 : 3400) : (rest ? 1536 : 2200);
    else if (!vec && !xi_out && broadcast && K >= 6) per_sm = K >= 8 ? 2600 : 1800;
    const int64_t quad_wave = (int64_t)ctx->n_sm * 4096, half_wave = (int64_t)ctx->n_sm * (broadcast ? 6400 : 4800);
    const bool shrt = d <= (int64_t)ctx->n_sm * per_sm || (!vec && many && (broadcast || !rest) && d > quad_wave && d <= half_wave);
    // By ticket when a fixed stride takes every block round many times; four blocks of either kernel fit an SM.
    // Measured, fixed stride and tickets, with broadcast: K = 20, d = 2.6M 71.6 and 72.7 us (two rounds); K = 30,
    // d = 7M 287 and 280 us (six); K = 60, d = 20M 1555 and 1524 us; K = 8, d = 198M 2179 and 2035 us (without broadcast
    // 1100 and 1019 us).  Rows at any alignment: K = 30, d = 7M 288 and 287 us (without broadcast 132 and 135 us), K = 60,
    // d = 20M 1804 and 1644 us.  Two quads per thread spilled at three blocks per SM: 2052 us at d = 198M.
    const bool tickets = !shrt && !xi_out && (d + 3) / 4 > (int64_t)ctx->n_sm * 8 * threads * (vec ? 4 : 8);
    int64_t blocks = ((shrt ? d : (d + 3) / 4) + threads - 1) / threads;
    const int64_t cap = (int64_t)ctx->n_sm * (!tickets ? 8 : 4);
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    unsigned int *ticket = ctx->combine_ticket + 1;
    if (shrt) {
        const cudaError_t e = fda_launch_dependent(xi_out ? k_average_short<true> : k_average_short<false>, (int)blocks, threads, 0, s,
                                                   w, row_stride, K, d, w_t0, gate, broadcast, xi_out, ctx->part_np);
        if (e != cudaSuccess || !xi_out) return e;
    } else {
        auto kern = xi_out    ? (vec ? k_average<true, false> : k_average_shifted<true, false>)
                    : tickets ? (vec ? k_average<false, true> : k_average_shifted<false, true>)
                              : (vec ? k_average<false, false> : k_average_shifted<false, false>);
        const cudaError_t e = fda_launch_dependent(kern, (int)blocks, threads, 0, s,
                                                   w, row_stride, K, d, w_t0, gate, broadcast, xi_out, ctx->part_np, ticket);
        if (e != cudaSuccess || !xi_out) return e;
    }
    return fda_launch_dependent(k_scale_xi, (int)blocks, threads, 0, s, xi_out, d, ctx->part_np, (int)blocks, gate);
}
