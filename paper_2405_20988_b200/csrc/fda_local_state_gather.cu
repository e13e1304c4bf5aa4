// Sketch pass over sorted per-cell lists (the main path of fda_local_state with a sketch).
//
// What the pass computes is stated in fda_local_state.cu (Section 3: drift and ||u||^2;
// Section 3.1: sk(u); Section 3.2: <xi,u>).  This file turns the scatter
// sk[i][h_i(j)] += s_i(j) u[j] into a gather: the bucket and sign of an index never change,
// so the context holds, for every tile of T indices, the indices of each sketch row sorted by
// cell and laid out as a program for a warp (the schedule of fda_sched.cu).  A lane keeps the
// sum of one cell in registers, walks the cell's list and reads the drifts it needs from a
// tile in shared memory; a cell of the bins is touched once per tile and list instead of once
// per update, with plain loads and stores, because a cell belongs to one list (cells that had
// to be cut into pieces are added atomically).  One update costs one 4-byte shared-memory read.
//
// A block serves a group of 4 workers and a strided set of tiles, with two kinds of warps:
//   producers  8 warps (5 when the walk is most of the work).  A thread owns four consecutive indices
//              of a batch (1024 indices with 8 warps; the last batch of a tile may be a part): it loads the four workers' values and w_t0
//              (xi) with 128-bit loads into registers (the landing zone: nothing else is staged),
//              subtracts, adds up ||u||^2 and <xi,u> (fp32 within a tile, fp64 across tiles) and
//              stores the four drifts of an index as one 16-byte row of the tile: ut[index][4].
//              The next batch is asked for as soon as the registers are free.  Measured on B200:
//              what a block streams from memory grows with the number of warps that have loads
//              in flight (4.6 TB/s with 8 warps per SM, 6.5 with 16, 7.0 with 24), not with the
//              loads a warp has in flight; deeper software pipelines here changed nothing, and
//              32-bit loads ran at a quarter of the speed;
//   walkers    20 warps (23).  They take the tile's items (32 lists, one per lane) from a counter,
//              longest first; per step a lane loads one 16-bit entry's row with a 128-bit load
//              (the schedule orders the entries so that the eight lanes of a pass through
//              shared memory hit eight different bank groups) and adds it with the entry's
//              sign; when the item ends the 32 sums are added to the bins.
// The tile is double buffered: while the walkers are on tile n the producers fill the other
// buffer with tile n + 1, and one block-wide barrier per tile hands the buffers over.  Nothing
// in this kernel waits on another block or spins on memory.
//
// What bounds it: the load/store unit's data pipe (74 % busy; 6.3 wavefronts per 128 updates
// are the floor of this design, 8.2 are spent).  The loads of the next tile's first batch are asked for in front of
// the barrier, and the sums of squares go through six shuffles instead of twenty (they take that pipe, too):
// with lanes that keep their cells 2065 -> 1876 us at 5 x 250, K = 8, d = 198M, 312 -> 285 at K = 30, d = 7M.  Between two items a walker has nothing to gather,
// so the way from item to item is kept short: the record's offset comes from shared memory (read
// from L2 after the barrier it stood in front of the first entries of every tile), the first item of
// a tile goes to a warp by its number, and the next item's number and descriptor are fetched before
// the walk of the current one.  5 x 250, K = 8, d = 198M: 2.44 -> 2.38 ms; K = 30, d = 7M: 372 -> 356 us;
// 7 x 500, K = 60, d = 20M: 2.98 -> 2.89 ms.  Fewer live registers (tile counts and indices in 32 bits,
// eight steps in one block of code) took them to 2.33 ms, 347 us and, with 5 + 23 warps, 2.57 ms.  Tried and slower: hand-over through mbarriers instead of
// the barrier (2.52 ms: the bins still need the walkers to meet between tiles, or two of them would
// add to one cell at a time), entries of the next item asked for before the flush (2.61 ms), 24
// walkers at 64 registers (2.40 ms).
//
// Lanes that keep their cells.  A bucket is a*j + b mod p mod m, a lattice: in a tile of thousands of consecutive
// indices nearly every cell has the same number of them (the variance of the counts is a tenth of that of random
// buckets; one row in twenty or so is an exception).  So lists need not be handed out by length: on long vectors
// every cell belongs to one lane of one walker warp for the whole launch.  What that saves: the sum of a cell
// lives in registers (the list of a tile is added up from zero and added to it once per tile, as to a bin before),
// so there are no bins, no flush with its conflicts, no counters and no item tables; a warp's program is known
// ahead, so the next eight steps are always asked for, across items and across the hand-over; walkers do not
// stop between items all at once.  The order of the cells of a row is chosen so that the lists of eight neighbours are
// copies of one another shifted by an odd number of indices (fda_sched.cu): as long as one another, and spread over
// the bank groups; steps per entry 1.12 at 5 x 250, 1.19 at 7 x 500 (list kernel 1.16 and 1.23).  Walkers 12 to 24
// of 28 to 32 warps (lane_walkers in fda_sched.cu); the others produce.  Measured, the
// list kernel and this one: 5 x 250, K = 8, d = 198M 2322 and 1860 us (2500 and 2218 us after half a second, at the
// power limit); K = 30, d = 7M 347 and 283; 7 x 500, K = 60, d = 20M 2560 and 2022; 8 x 1000, K = 20, d = 2.6M 203 and
// 166; K = 8, d = 20M: 1 x 250 181 and 128, 3 x 500 218 and 173, 4 x 1000 394 and 241.  The gain depends on the hash (steps
// per entry) and on the clock: 7 x 500, K = 60 came to 12 to 25 % on different GPUs.
//
// Its line: states without a projection, blocks of more than four tiles.  Measured with the finalize kernel, list kernel and
// this one, by tiles a block: 5 x 250, K = 14, d = 1.2M (5.2) 38.2 and 34.9 us, K = 16, d = 1.6M (7) 44.8 and 40.0, K = 30, d = 0.7M
// (6.3) 43.8 and 39.8; 3 x 100, K = 10, d = 1.5M (6) 28.5 and 25.8; 7 x 500, K = 44, d = 0.6M (7.9) 72.5 and 62.9, K = 20, d = 1M
// (5.6) 54.7 and 50.8; 4 x 1000, K = 20, d = 1M (4.8) 60.0 and 43.4; 8 x 1000, K = 26, d = 0.3M (4.6) 47.2 and 42.2, K = 44, d = 0.3M
// (6.8) 63 and 54.  That pays for the second schedule (0.6 to 1 ms of fda_create) after some 200 steps.  Shorter vectors gain
// less (5 x 250, K = 10, d = 1.2M, four tiles: 28.7 and 27.0).  With xi the list kernel stays, a
// fifth slower on long vectors: what it gives is one order of additions for all sizes, so the digits of a run that projects do
// not depend on which side of the line its vectors are.  That order shows right after a synchronisation, when the mean
// drift is the rounding of the average itself: the row norms of S-bar then differ from the fourth digit on.  They are
// rounding noise on either kernel (the cells are equally far from 64 bits, 1.2e-7 of their norm); runs without a projection
// took the other order, and the speed.
//
// fda_mean_state_gather.cu holds the sibling of this kernel that computes the averaged state of
// fda_mean_state from the list schedule.

#include <algorithm>

#include "fda_internal.h"
#include "fda_worker_kernel.cuh"

// One launch of the kernel whose lanes keep their cells, with `walkers` warps that walk (blocks == 0: only sets its
// shared-memory limit).
static cudaError_t fda_lanes_run(int walkers, bool parts, const fda_list::ListParams &p, int blocks, bool dependent, cudaStream_t s)
{
    if (parts) return fda_lanes_22(p, blocks, dependent, s);
    switch (walkers) {
        case 12: return fda_lanes_12(p, blocks, dependent, s);
        case 16: return fda_lanes_16(p, blocks, dependent, s);
        case 20: return fda_lanes_20(p, blocks, dependent, s);
        case 23: return fda_lanes_23(p, blocks, dependent, s);
        default: return fda_lanes_24(p, blocks, dependent, s);
    }
}

namespace {

using namespace fda_list;

constexpr int kShortWarps = 24;
constexpr int kShortChunks = 2;                // chunks of 128 indices a warp forms: tiles of up to 6144 indices
constexpr uint32_t kShortBins = kShortWarps * GW * 2 * 8;      // offset of the bins, behind the warps' sums
inline size_t short_smem_bytes(int lm, int T) { return kShortBins + (size_t)lm * GW * 4 + (size_t)(T + kListPadRows) * GW * 4; }

// The sketch pass of vectors with so few tiles that no block has more than one: p.part_tiles blocks (one
// to three) share a tile - all of them form its drifts, each walks every p.part_tiles-th item - and their
// bins, which differ in the cells they touch, are partial sums like those of any other blocks, so the
// cells come out the same bit for bit.
// Bound: latency, so there are no roles and no second buffer: every warp has its first item's entries
// on their way (the schedule is older than the kernel before this one, so even in front of
// fda_grid_wait), then all the loads of its two chunks of indices, stores the drifts, and after one barrier walks.
// Measured, 5 x 250, K = 5, d = 61,706, with its finalize kernel, back to back: 8.7 us with up to three blocks
// to a tile (8.9 with two or four), against 10.3 with 16 producer and 12 walker warps on shared tiles and
// 14.4 with 8 + 20 warps on a tile of its own.
template <bool LINEAR, bool VEC>
__global__ void __launch_bounds__(kShortWarps * 32, 1) k_local_state_short(const ListParams p)
{
    constexpr int kThreads = kShortWarps * 32;
    constexpr int kAhead = 7;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int split = p.part_tiles, sub = (int)blockIdx.x / (p.groups * p.cpg), blk = (int)blockIdx.x % (p.groups * p.cpg);
    const int g = blk % p.groups, c = blk / p.groups;         // the block's tile is tile c
    const int T = p.T, lm = p.l * p.m;
    const uint32_t smem_base = (uint32_t)__cvta_generic_to_shared(smem_raw);
    const uint32_t base = smem_base + kShortBins + (uint32_t)lm * 16u;
    double *sums = reinterpret_cast<double *>(smem_raw);
    float *bins = reinterpret_cast<float *>(smem_raw + kShortBins);

    const unsigned char *rec = p.sched + load_u64(p.sched_off + c);
    const uint32_t *tab = reinterpret_cast<const uint32_t *>(rec);
    int it = warp * split + sub;
    const int n_items = (int)__ldg(tab);
    const uint16_t *cells = reinterpret_cast<const uint16_t *>(rec + fda_sched_cells_off(n_items));
    const unsigned char *ent0 = rec + fda_sched_entries_off(n_items);
    int steps = 0;
    uint32_t cell = 0;
    const uint2 *ent = nullptr;
    uint2 ch[kAhead];
    auto fetch = [&]() {
        const uint32_t d0 = __ldg(tab + 4 + 2 * it), chunk0 = __ldg(tab + 5 + 2 * it);
        steps = (int)(d0 & 0xffffu);
        cell = __ldg(cells + (size_t)(d0 >> 16) * kListSlots + lane);
        ent = reinterpret_cast<const uint2 *>(ent0 + (size_t)chunk0 * 256) + lane;
#pragma unroll
        for (int q = 0; q < kAhead; ++q)
            if (4 * q < steps) ch[q] = __ldg(ent + (size_t)q * kListSlots);
    };
    if (it < n_items) fetch();
    for (int t = tid; t < lm * GW; t += kThreads) bins[t] = 0.f;
    if (tid < kListPadRows) store_row(base + (uint32_t)(T + tid) * 16u, 0.f, 0.f, 0.f, 0.f);
    fda_grid_wait();

    form_drifts<LINEAR, VEC, kShortChunks>(p, g, (int64_t)c * T, warp, kShortWarps, base, sums + warp * GW * 2);
    __syncthreads();

    // ---- items warp * split + sub, then every (kShortWarps * split)-th ----
    while (it < n_items) {
        unsigned long long a01 = 0ull, a23 = 0ull;
#pragma unroll
        for (int q = 0; q < kAhead; ++q) walk_chunk(ch[q], steps - 4 * q, base, a01, a23);
        for (int c0 = kAhead; 4 * c0 < steps; ++c0)
            walk_chunk(__ldg(ent + (size_t)c0 * kListSlots), steps - 4 * c0, base, a01, a23);
        const uint32_t done = cell;
        it += kShortWarps * split;
        if (it < n_items) fetch();
        flush_item(bins, lm, done, a01, a23);
    }
    __syncthreads();

    float *out = p.part_sk + (size_t)blockIdx.x * (size_t)lm * GW;
    for (int t = tid; t < lm; t += kThreads) reinterpret_cast<float4 *>(out)[t] = reinterpret_cast<const float4 *>(bins)[t];
    if (tid < GW * 2) {
        double t = 0.0;
        if (sub == 0)
            for (int q = 0; q < kShortWarps; ++q) t += sums[q * GW * 2 + tid];
        p.part_np[(size_t)blockIdx.x * GW * 2 + tid] = t;
    }
}

// The partial sums of a call come from up to three launches of the kernel (the main one and the
// two that fill the SMs it leaves idle, see fda_launch_local_state_gather): launch q served the
// groups g_first .. g_first + groups - 1 with cpg blocks each, block c * groups + (g - g_first)
// writing slot slot_base + that number.
struct ListParts {
    int n;
    int slot_base[3], g_first[3], groups[3], cpg[3];
};

// states[k][.] = sum of the partials of worker k's blocks in fp64, in a fixed order: four
// adjacent lanes share one output, lane s adds the blocks s, s + 4, ... of the worker's group in
// each launch in order, and the four sums are added as (s0 + s1) + (s2 + s3).
// Bound: latency (a few megabytes at most, from L2): a lane asks for kLoads values at a time - four, eight
// or twelve, as few as cover the blocks of a group in one or two rounds - and blockIdx.y is the worker
// group, so that no index is divided.
// Measured with the kernel before it, 5 x 250, K = 10, d = 150K (25 blocks a group): 12.1 us with eight or sixteen
// values at a time and 64-bit divisions, 11.7 now; four at a time cost 3 us there, and twelve cost 7 us at
// 7 x 500, K = 60 (9 blocks a group).
template <int kLoads>
__global__ void __launch_bounds__(256) k_finalize_gather(const ListParams p, const ListParts parts, uint32_t flags, float *__restrict__ states)
{
    const int lm = p.l * p.m, slen = 2 + lm * (p.groups / p.wgroups);       // lm: cells of a part
    const int t = blockIdx.x * 256 + threadIdx.x, sub = t & 3, kl = (t >> 2) % GW, e = t / (4 * GW), g = blockIdx.y;
    const bool on = e >= slen ? false
                  : e == 0    ? (flags & FDA_STATE_NORM) != 0
                  : e == 1    ? (flags & FDA_STATE_LINEAR) != 0 && p.have_xi != 0
                              : (flags & FDA_STATE_SKETCH) != 0;
    const int part = e < 2 ? 0 : (e - 2) / lm;                  // part 0 also has the norm and the projection
    fda_grid_wait();
    double acc = 0.0;
    for (int q = 0; q < parts.n; ++q) {
        const int gl = part * p.wgroups + g - parts.g_first[q];
        if (!on || gl < 0 || gl >= parts.groups[q]) continue;
        const int nb = parts.cpg[q];                            // blocks of this group: gl, gl + groups, ...
        const size_t first = (size_t)(parts.slot_base[q] + gl), step = (size_t)parts.groups[q];
        const double *np = p.part_np + (first * GW + kl) * 2 + e;
        const float *sk = p.part_sk + first * lm * GW + (size_t)(e - 2 - part * lm) * GW + kl;
        if (e < 2) {
            for (int j = sub; j < nb; j += 4 * kLoads) {
                double v[kLoads];
#pragma unroll
                for (int u = 0; u < kLoads; ++u) v[u] = np[(size_t)(j + 4 * u < nb ? j + 4 * u : j) * step * GW * 2];
#pragma unroll
                for (int u = 0; u < kLoads; ++u) acc += j + 4 * u < nb ? v[u] : 0.0;
            }
        } else {
            for (int j = sub; j < nb; j += 4 * kLoads) {
                float v[kLoads];
#pragma unroll
                for (int u = 0; u < kLoads; ++u) v[u] = sk[(size_t)(j + 4 * u < nb ? j + 4 * u : j) * step * lm * GW];
#pragma unroll
                for (int u = 0; u < kLoads; ++u) acc += j + 4 * u < nb ? (double)v[u] : 0.0;
            }
        }
    }
    const double pair = acc + __shfl_xor_sync(0xffffffffu, acc, 1);      // lanes 0,1: s0 + s1; lanes 2,3: s2 + s3
    const double other = __shfl_xor_sync(0xffffffffu, pair, 2);
    const int k = g * GW + kl;
    if (e < slen && sub == 0 && k < p.K) states[(size_t)k * slen + e] = (float)(pair + other);
}

// The same sums with the four workers of the group in each lane, 128-bit loads of the partials: a quarter of
// the threads, for launches whose threads would not all be resident at once.  Lane s stores worker s.
template <int kLoads>
__global__ void __launch_bounds__(256) k_finalize_gather_wide(const ListParams p, const ListParts parts, uint32_t flags, float *__restrict__ states)
{
    const int lm = p.l * p.m, slen = 2 + lm * (p.groups / p.wgroups);
    const int t = blockIdx.x * 256 + threadIdx.x, sub = t & 3, e = t / 4, g = blockIdx.y;
    const bool on = e >= slen ? false
                  : e == 0    ? (flags & FDA_STATE_NORM) != 0
                  : e == 1    ? (flags & FDA_STATE_LINEAR) != 0 && p.have_xi != 0
                              : (flags & FDA_STATE_SKETCH) != 0;
    const int part = e < 2 ? 0 : (e - 2) / lm;
    fda_grid_wait();
    double acc[GW] = {};
    for (int q = 0; q < parts.n; ++q) {
        const int gl = part * p.wgroups + g - parts.g_first[q];
        if (!on || gl < 0 || gl >= parts.groups[q]) continue;
        const int nb = parts.cpg[q];
        const size_t first = (size_t)(parts.slot_base[q] + gl), step = (size_t)parts.groups[q];
        if (e < 2) {
            const double *np = p.part_np + first * GW * 2 + e;
            for (int j = sub; j < nb; j += 4)
#pragma unroll
                for (int k = 0; k < GW; ++k) acc[k] += np[(size_t)j * step * GW * 2 + 2 * k];
        } else {
            const float4 *sk = reinterpret_cast<const float4 *>(p.part_sk) + first * lm + (e - 2 - part * lm);
            for (int j = sub; j < nb; j += 4 * kLoads) {
                float4 v[kLoads];
#pragma unroll
                for (int u = 0; u < kLoads; ++u) v[u] = sk[(size_t)(j + 4 * u < nb ? j + 4 * u : j) * step * lm];
#pragma unroll
                for (int u = 0; u < kLoads; ++u) {
                    const bool in = j + 4 * u < nb;
                    acc[0] += in ? (double)v[u].x : 0.0;
                    acc[1] += in ? (double)v[u].y : 0.0;
                    acc[2] += in ? (double)v[u].z : 0.0;
                    acc[3] += in ? (double)v[u].w : 0.0;
                }
            }
        }
    }
    double mine = 0.0;
#pragma unroll
    for (int k = 0; k < GW; ++k) {
        const double pair = acc[k] + __shfl_xor_sync(0xffffffffu, acc[k], 1);
        const double other = __shfl_xor_sync(0xffffffffu, pair, 2);
        if (sub == k) mine = pair + other;
    }
    const int k = g * GW + sub;
    if (e < slen && k < p.K) states[(size_t)k * slen + e] = (float)mine;
}

void (*pick_short(bool linear, bool vec))(ListParams)
{
    if (linear) return vec ? k_local_state_short<true, true> : k_local_state_short<true, false>;
    return vec ? k_local_state_short<false, true> : k_local_state_short<false, false>;
}

template <int PW, int WW, bool PARTS>
cudaError_t launch_lists(ListParams &p, int blocks, size_t smem, bool dependent, cudaStream_t s)
{
    if (p.T % 128 != 0 || p.T < PW * 128 || PW * 32 * 16 < p.tab_bytes) return cudaErrorNotSupported;
    // all warps form the first tile when a block has at most twelve.  Measured, kernel and finalize back to back:
    // 5 x 250, K = 20, d = 300,000 (two tiles) 18.3 -> 17.4 us, K = 10, d = 1.2M (four) 34.1 -> 32.4 us; 7 x 500, K = 10,
    // d = 1.2M (five) 46.0 -> 44.5 us; K = 20, d = 2M (twelve) 75.7 -> 75.3 us.  Rows in parts: 8 x 1000, K = 20, d = 160K
    // 26.2 -> 25.7 us, K = 40, d = 100K 28.4 -> 27.8 (with xi not: the norms' order of additions stays).
    const bool first = !(PARTS && p.have_xi) && p.tiles <= 12 * (int64_t)p.cpg;
    auto kern = first ? pick_kernel<PW, WW, PARTS, true, 0>(p.have_xi != 0, p.vec != 0)
                      : pick_kernel<PW, WW, PARTS, false, 0>(p.have_xi != 0, p.vec != 0);
    if (dependent) return fda_launch_dependent(kern, blocks, (PW + WW) * 32, smem, s, p);
    kern<<<blocks, (PW + WW) * 32, smem, s>>>(p);
    return cudaGetLastError();
}

}  // namespace

// The kernels' dynamic shared memory limit, set once per context (on the context's device).
cudaError_t fda_setup_local_state_gather(const fda_ctx *ctx)
{
    if (ctx->lane_prog) {
        ListParams p{};
        p.lane_items = ctx->lane_items; p.T = ctx->lane_T;
        for (p.vec = 0; p.vec < 2; ++p.vec) {
            const cudaError_t e = fda_lanes_run(ctx->lane_walkers, ctx->lane_parts > 1, p, 0, false, nullptr);
            if (e != cudaSuccess) return e;
        }
    }
    for (int i = 0; i < 4; ++i) {
        const bool linear = i & 1, vec = i & 2;
        for (auto kern : {pick_kernel<8, 20, false, false, 0>(linear, vec), pick_kernel<5, 23, false, false, 0>(linear, vec),
                          pick_kernel<8, 20, false, true, 0>(linear, vec), pick_kernel<5, 23, false, true, 0>(linear, vec),
                          pick_kernel<8, 20, true, false, 0>(linear, vec), pick_kernel<8, 20, true, true, 0>(false, vec), pick_short(linear, vec)}) {
            const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ctx->smem_optin);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

// Returns cudaErrorNotSupported when the request does not fit this path (the caller then uses
// the other kernels); any other value is the result of the launches.
cudaError_t fda_launch_local_state_gather(fda_ctx *ctx, const float *w, int64_t row_stride, int K,
                                          int64_t d, const float *w_t0, const float *xi,
                                          uint32_t flags, float *states, cudaStream_t s)
{
    if (!(flags & FDA_STATE_SKETCH) || ctx->l == 0 || !ctx->sched) return cudaErrorNotSupported;
    const float *xi_used = (flags & FDA_STATE_LINEAR) ? xi : nullptr;

    ListParams p{};
    p.w = w; p.w_t0 = w_t0; p.xi = xi_used; p.row_stride = row_stride;
    p.K = K; p.d = d; p.have_xi = xi_used != nullptr;
    p.vec = ((((uintptr_t)w | (uintptr_t)w_t0 | (uintptr_t)(xi_used ? xi_used : w)) & 15u) == 0) && (row_stride % 4 == 0);
    const int wgroups = (K + GW - 1) / GW;
    const bool lanes = ctx->lane_prog && !xi_used && fda_lanes_pay((d + ctx->lane_T - 1) / ctx->lane_T, wgroups * ctx->lane_parts, ctx->n_sm);
    const int sched_parts = lanes ? ctx->lane_parts : ctx->sched_parts;
    p.l = ctx->l / sched_parts; p.m = ctx->m;
    p.part_tiles = (int)(lanes ? ctx->lane_tiles : ctx->sched_tiles);
    p.T = lanes ? ctx->lane_T : ctx->sched_T;
    p.sched = lanes ? ctx->lane_sched : ctx->sched; p.sched_off = lanes ? ctx->lane_off : ctx->sched_off;
    if (lanes) { p.lane_prog = ctx->lane_prog; p.lane_rows = ctx->lane_rows; p.lane_items = ctx->lane_items; }
    p.part_sk = ctx->part_sk; p.part_np = ctx->part_np;
    p.tiles = (d + p.T - 1) / p.T;
    p.tab_bytes = fda_list_table_bytes(ctx->sched_ni_max);
    p.wgroups = wgroups;
    p.groups = wgroups * sched_parts;
    if (p.groups > ctx->n_sm) return cudaErrorNotSupported;
    int64_t cpg = ctx->n_sm / p.groups;
    if (cpg > p.tiles) cpg = p.tiles;
    p.cpg = (int)cpg;
    const int blocks = p.groups * p.cpg, lm = p.l * p.m;
    if ((size_t)blocks * lm * GW > ctx->part_sk_floats || blocks > ctx->max_blocks ||
        (size_t)blocks * GW * 2 > ctx->part_np_doubles)
        return cudaErrorNotSupported;
    const size_t smem = fda_list_smem_bytes(p.l, p.m, p.T, ctx->sched_ni_max);
    if (!lanes && smem > (size_t)ctx->smem_optin) return cudaErrorNotSupported;

    // A vector with at most one tile per block runs on k_local_state_short, whose tiles hold up to 6144 indices:
    // several blocks share a tile while the SMs last, and sketches of up to six rows stay with it when they do not.
    // Measured with the finalize kernel, back to back, d at 75 to 148 blocks of one tile, the short kernel against the
    // one with roles: 5 x 250, K = 10, d = 154K 10.5 and 11.4 us, K = 5, d = 455K 11.5 and 12.3; 3 x 200, K = 10,
    // d = 154K 9.5 and 11.0; 6 x 400, K = 10, d = 128K 13.0 and 13.7; but 7 x 500, K = 10, d = 128K 15.0 and 14.8,
    // 8 x 250 15.0 and 14.3, 16 x 100 21.6 and 20.8, where the walk is most of the work and 28 warps are better than 24.  With
    // blocks to share the tiles: 7 x 500, K = 10, d = 123K 13.4 and 14.8, 16 x 100, d = 147K 17.5 and 20.7.
    int split = 1;
    bool one_tile = false;
    if (sched_parts == 1) {
        if (!lanes && p.tiles == p.cpg && p.T <= kShortWarps * 128 * kShortChunks) {
            split = std::min(3, ctx->n_sm / blocks);
            one_tile = split > 1 || p.l <= 6;
        }
        p.part_tiles = split;
    }
    // 8 producer + 20 walker warps, or 5 + 23 when a loaded index pays for more walking: l steps, and its share of the
    // starts and flushes of the lists, which cost about ten steps each (T / m indices to a list and row).  Measured, 8 + 20
    // and 5 + 23, K = 8, d = 20M, by l * (1 + 10 * m / T): 7.4 (5 x 300) 257 and 311 us; 9.9 (5 x 500) 311 and
    // 313, (7 x 250) 300 and 329; 10.1 (6 x 350) 330 and 322; 10.9 (5 x 600) 348 and 317; 11.9 (6 x 500) 367 and 332; 13.8
    // (7 x 500) 421 and 355; from eight rows on 5 + 23 whatever the lists (8 x 100, 9.3: 406 and 376; 8 x 250 346 and 340;
    // 9 x 250 397 both; 12 x 250 495 and 500; 16 x 100 757 and 695).  Other splits: 7 x 500, K = 60, d = 20M: 2.76 ms
    // with 5 + 23, 2.90 with 4 + 24, 2.95 with 8 + 20, 2.68 against 2.64 with 6 + 22; 5 x 250, K = 8, d = 198M: 2.35 ms
    // with 8 + 20, 2.46 with 7 + 21, 2.48 with 9 + 19, 2.61 with 12 + 16; 8 x 1000 in parts, K = 20, d = 2.6M: 214 us with
    // 8 + 20, 216 with 10 + 18, 231 with 6 + 22, 226 with 8 + 24 (64 registers).
    const bool walking = p.l >= 8 || (int64_t)p.l * (p.T + 10 * p.m) >= 10 * (int64_t)p.T;
    auto launch = [&](ListParams &q, int grid, cudaStream_t st, bool dependent) {
        if (lanes) return fda_lanes_run(ctx->lane_walkers, sched_parts > 1, q, grid, dependent, st);
        if (sched_parts > 1) return launch_lists<8, 20, true>(q, grid, smem, dependent, st);
        if (one_tile)
            return fda_launch_dependent(pick_short(q.have_xi != 0, q.vec != 0), grid, kShortWarps * 32,
                                        short_smem_bytes(q.l * q.m, q.T), st, q);
        return walking ? launch_lists<5, 23, false>(q, grid, smem, dependent, st)
                        : launch_lists<8, 20, false>(q, grid, smem, dependent, st);
    };
    ListParts parts{};
    parts.n = 1;
    parts.slot_base[0] = 0; parts.g_first[0] = 0; parts.groups[0] = p.groups; parts.cpg[0] = p.cpg * split;

    // When the groups do not divide the SMs (K = 60: 15 groups x 9 blocks on 148 SMs) the SMs left
    // over get the last tiles of every group, from the same kernel launched on a second stream with
    // shifted pointers: first one block for each of the first `extra` groups, then the other groups
    // on as many blocks each as fit.  The main launch stops at tile t1; all launches write their own
    // slots of the partial sums.  Taken when the second of those launches still has a block per group
    // and the job is long enough for the gain (tiles / cpg against t1 / cpg tile walks) to show: where a block saves more than two
    // walks, from 36 tiles a block on with lanes that keep their cells.  Measured, K = 60, one launch and three, by tiles a
    // block: 3 x 100 32: 133.6 and 134.7 us, 36: 148.0 and 140.8; 5 x 250 40: 186.8 and 185.7, 48: 219.6 and 214.5; 7 x 500 40: 260.4 and
    // 253.6, 48: 307.8 and 296.5; 8 x 250 40: 271.0 and 257.5; 1 x 250 40: 115.2 and 116.2, 44: 125.4 and 122.4.  The other kernel would
    // gain from 40 on (5 x 250 221.7 and 214.4, 7 x 500 322.9 and 306.5) but keeps 64 and with it the order of its additions.
    const int extra = ctx->n_sm - blocks;
    const int rest = p.groups - extra;                         // groups of the second tail launch (extra < groups)
    int64_t t1 = p.tiles;
    int cpg_b = 0;
    if (sched_parts == 1 && extra > 0 && rest > 0 && extra / rest >= 1 && ctx->side_stream && p.tiles >= (lanes ? 36 : 64) * (int64_t)p.cpg) {
        cpg_b = extra / rest;
        // tail walks per block: n_tail + n_tail / cpg_b; main walks per block: (tiles - n_tail) / cpg
        const double per_tail = 1.0 + 1.0 / (double)cpg_b;
        int64_t n_tail = (int64_t)((double)p.tiles / (1.0 + (double)p.cpg * per_tail));
        n_tail = n_tail / cpg_b * cpg_b;
        const int64_t main_walks = (p.tiles - n_tail + p.cpg - 1) / p.cpg;
        const size_t slots = (size_t)blocks + extra + (size_t)rest * cpg_b;
        if (n_tail >= 4 * cpg_b && main_walks + 2 < (p.tiles + p.cpg - 1) / p.cpg &&
            slots * lm * GW <= ctx->part_sk_floats && slots * GW * 2 <= ctx->part_np_doubles)
            t1 = p.tiles - n_tail;
    }
    cudaError_t e;
    if (t1 < p.tiles) {
        const int64_t shift = t1 * p.T;                        // elements in front of the tail (a multiple of 1024)
        ListParams ta = p;
        ta.w = p.w + shift; ta.w_t0 = p.w_t0 + shift; ta.xi = p.xi ? p.xi + shift : nullptr;
        ta.d = p.d - shift; ta.tiles = p.tiles - t1; ta.sched_off = p.sched_off + t1;
        if (p.lane_prog) ta.lane_prog = p.lane_prog + (size_t)t1 * (p.lane_items + 1);
        ListParams tb = ta;
        ta.K = extra * GW; ta.groups = ta.wgroups = extra; ta.cpg = 1;
        ta.part_sk = p.part_sk + (size_t)blocks * lm * GW; ta.part_np = p.part_np + (size_t)blocks * GW * 2;
        tb.w = ta.w + (size_t)extra * GW * (size_t)row_stride; tb.K = K - extra * GW; tb.groups = tb.wgroups = rest; tb.cpg = cpg_b;
        tb.part_sk = ta.part_sk + (size_t)extra * lm * GW; tb.part_np = ta.part_np + (size_t)extra * GW * 2;
        parts.n = 3;
        parts.slot_base[1] = blocks; parts.g_first[1] = 0; parts.groups[1] = extra; parts.cpg[1] = 1;
        parts.slot_base[2] = blocks + extra; parts.g_first[2] = extra; parts.groups[2] = rest; parts.cpg[2] = cpg_b;
        ListParams main = p;
        main.tiles = t1; main.d = shift;
        e = cudaEventRecord(ctx->ev_fork, s);                  // (launches that events order are ordinary ones)
        if (e == cudaSuccess) e = cudaStreamWaitEvent(ctx->side_stream, ctx->ev_fork, 0);
        if (e == cudaSuccess) e = launch(ta, extra, ctx->side_stream, false);
        if (e == cudaSuccess) e = launch(tb, rest * cpg_b, ctx->side_stream, false);
        if (e == cudaSuccess) e = cudaEventRecord(ctx->ev_join, ctx->side_stream);
        if (e == cudaSuccess) e = launch(main, blocks, s, false);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, ctx->ev_join, 0);
    } else {
        e = launch(p, blocks * split, s, true);
    }
    if (e != cudaSuccess) return e;
    ctx->last_ls_launches = parts.n + 1;
    ctx->last_schedule = lanes ? 2 : 1;
    const int nb = parts.cpg[0];
    // one worker per lane while all those threads are resident at once (2048 to an SM), four beyond that.  Measured,
    // kernel and finalize back to back, one and four per lane: 5 x 250, K = 10, d = 1.2M (60K threads) 30.0 and 34.3 us;
    // 5 x 250, K = 30, d = 2M (160K) 110.6 both; 7 x 500, K = 60, d = 1.2M (841K) 191.0 and 184.7 us; 8 x 1000,
    // K = 30, d = 300,000 (1.02M) 55.7 and 48.0 us.
    const int64_t sums = (int64_t)(2 + ctx->lm) * 4;
    const bool wide = sums * GW * p.wgroups > (int64_t)ctx->n_sm * 2048;
    auto fin = wide ? (nb <= 16 ? k_finalize_gather_wide<4> : nb <= 32 ? k_finalize_gather_wide<8> : k_finalize_gather_wide<12>)
                    : (nb <= 16 ? k_finalize_gather<4> : nb <= 32 ? k_finalize_gather<8> : k_finalize_gather<12>);
    const dim3 fb((unsigned)((sums * (wide ? 1 : GW) + 255) / 256), (unsigned)p.wgroups);
    if (parts.n == 1) return fda_launch_dependent(fin, fb, 256, 0, s, p, parts, flags, states);
    fin<<<fb, 256, 0, s>>>(p, parts, flags, states);       // waits for an event too: an ordinary launch
    return cudaGetLastError();
}
