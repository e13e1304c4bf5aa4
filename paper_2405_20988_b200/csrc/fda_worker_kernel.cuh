// The sketch pass over the list schedule with producer and walker warps: k_local_state_gather, which
// fda_local_state_gather.cu describes and launches.  The variants whose lanes keep their cells are
// instantiated in fda_lanes_*.cu, a file for each number of walker warps.
#ifndef FDA_WORKER_KERNEL_CUH_
#define FDA_WORKER_KERNEL_CUH_

#include "fda_internal.h"
#include "fda_list_kernel.cuh"

cudaError_t fda_lanes_12(const fda_list::ListParams &p, int blocks, bool dependent, cudaStream_t s);
cudaError_t fda_lanes_16(const fda_list::ListParams &p, int blocks, bool dependent, cudaStream_t s);
cudaError_t fda_lanes_20(const fda_list::ListParams &p, int blocks, bool dependent, cudaStream_t s);
cudaError_t fda_lanes_22(const fda_list::ListParams &p, int blocks, bool dependent, cudaStream_t s);   // sketch rows in parts
cudaError_t fda_lanes_23(const fda_list::ListParams &p, int blocks, bool dependent, cudaStream_t s);
cudaError_t fda_lanes_24(const fda_list::ListParams &p, int blocks, bool dependent, cudaStream_t s);

namespace {

using namespace fda_list;

// Sums of the four workers' values over the warp: the sum of v[lane >> 3] comes back.  Every step halves the
// values of a lane, so six shuffles do what twenty would (a shuffle takes the load/store unit's time), in the same
// tree.
__device__ __forceinline__ float warp_sums(const float (&v)[GW])
{
    const bool hi = threadIdx.x & 16, odd = threadIdx.x & 8;
    const float a = (hi ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[2], 16);
    const float b = (hi ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, hi ? v[1] : v[3], 16);
    float t = (odd ? b : a) + __shfl_xor_sync(0xffffffffu, odd ? a : b, 8);
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    return t;
}

// The drifts of the chunks first, first + step, ... (CHUNKS of them at a time) of 128 indices of the tile
// that starts at index j0: all loads before any use, rows into the buffer at `base`, the warp's sums
// of squares and products with xi (fp32) into sums[8] (fp64, lane 0).  VEC: a lane owns four consecutive
// indices of a chunk, else the four indices lane, lane + 32, ...  Workers past K alias the group's
// first row: their sums are never written out.
template <bool LINEAR, bool VEC, int CHUNKS>
__device__ __forceinline__ void form_drifts(const ListParams &p, int g, int64_t j0, int first, int step, uint32_t base,
                                            double *sums)
{
    const int lane = threadIdx.x & 31, T = p.T;
    const float *wbase = p.w + (size_t)(g * GW) * (size_t)p.row_stride;
    float nf[GW], pf[GW];
#pragma unroll
    for (int k = 0; k < GW; ++k) { nf[k] = 0.f; pf[k] = 0.f; }
#pragma unroll 1
    for (int c0 = first; c0 < T / 128; c0 += step * CHUNKS) {
        float4 wv[CHUNKS][GW], w0v[CHUNKS], xv[CHUNKS];
#pragma unroll
        for (int b = 0; b < CHUNKS; ++b) {
            const int r = 128 * (c0 + step * b);
            const int64_t j = j0 + r + (VEC ? 4 * lane : lane), left = r < T ? p.d - j : 0;
            const int n = VEC ? (left >= 4 ? 4 : left > 0 ? (int)left : 0) : (left > 96 ? 4 : left > 0 ? (int)(left + 31) / 32 : 0);
            auto load = [&](const float *ptr) { return VEC ? load_quad<false>(ptr, n == 4, n) : load_strided(ptr, n); };
#pragma unroll
            for (int k = 0; k < GW; ++k) wv[b][k] = load(wbase + (g * GW + k < p.K ? (int64_t)k * p.row_stride : 0) + j);
            w0v[b] = load(p.w_t0 + j);
            if (LINEAR) xv[b] = load(p.xi + j);
        }
#pragma unroll
        for (int b = 0; b < CHUNKS; ++b) {
            const uint32_t r0 = 128u * (uint32_t)(c0 + step * b);
            if (r0 >= (uint32_t)T) break;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float w0 = comp(w0v[b], q);
                float u[GW];
#pragma unroll
                for (int k = 0; k < GW; ++k) {
                    u[k] = comp(wv[b][k], q) - w0;
                    nf[k] = fmaf(u[k], u[k], nf[k]);
                    if (LINEAR) pf[k] = fmaf(comp(xv[b], q), u[k], pf[k]);
                }
                const uint32_t r = r0 + (VEC ? 4u * lane + q : (uint32_t)lane + 32u * q);
                store_row(base + fda_list_row(r) * 16u, u[0], u[1], u[2], u[3]);
            }
        }
        if (CHUNKS > 1) break;                                 // (the caller has checked that one round covers the tile)
    }
    const float a = warp_sums(nf), b = LINEAR ? warp_sums(pf) : 0.f;
    if ((lane & 7) == 0) { sums[lane >> 2] = (double)a; sums[(lane >> 2) + 1] = (double)b; }
}

// Chunks of entries (four steps each) that a walker whose lanes keep their cells has on their way: four while the block
// has few walkers, each with one or two items, two beyond that.  Measured, us with two and four, K = 8, d = 20M: 2 x 250 168 and
// 140, 3 x 250 181 and 159, 3 x 100 194 and 179, 4 x 250 191 and 183, but with 20 and more walkers 5 x 250, d = 198M 1860
// and 1894, 7 x 500, K = 60 2022 and 2135, 8 x 1000, K = 20, d = 2.6M 165 and 177 (registers).
template <int WW>
constexpr int kLaneAhead = WW <= 16 ? 4 : 2;
constexpr uint32_t kLaneTiles = 2176;          // offset of the tile buffers when lanes keep their cells: behind the head, on a 128-byte boundary
inline size_t lane_smem_bytes(int T) { return kLaneTiles + 2 * (size_t)(T + kListPadRows) * GW * 4; }

// Shared-memory plan (bytes from the start of dynamic shared memory):
//   [0, 8)    item counters of the two tile buffers
//   [16, 48)  offsets of the schedule records of the tiles n, n + 1 (slot n mod 4)
//   [64, 2112) sums[warp][worker][2] (fp64): ||u||^2 and <xi,u>, of the producers over the tiles so far, of
//             the walkers (FIRST) over their part of the first tile
//   [2112, ..) two item tables (tab_bytes each): the head of a tile's schedule record
//   then      bins[l*m][4]
//   then      ut[2][T + 8][4]   (drift tiles, index-major; eight zero rows behind each)
// PW producer warps and WW walker warps: the split that is fastest depends on how much walking a
// loaded index pays for (l updates per worker).  PARTS: the sketch rows are in several parts with
// records of their own, and a block serves one part of one worker group.
// Measured: 8 x 1000 as two parts, K = 20, d = 2.6M: 212 us, against 510 us on the compare-and-swap
// kernel that served it before.
// VEC: w, w_t0 and xi are 16-byte aligned.  If not, a producer thread owns the four indices lane, lane + 32,
// ... of its warp's 128 instead of four consecutive ones, so that its 32-bit loads are coalesced (K = 30,
// d = 6,964,106 at a pitch of d: 529 -> 370 us; 7 x 500, K = 60, d = 20M: 4.38 -> 2.75 ms).
// FIRST: all warps form the first tile.  As the producers' own job it is a chain of round trips with nothing to
// walk meanwhile, which counts when a block has few tiles; the code for it costs long runs 1 %.
// LANES: cells stay with their lanes, at most LANES items to a walker warp (0: they do not).  Shared memory then
// holds the head and, from kLaneTiles on, the two tiles.
template <bool LINEAR, int PW, int WW, bool PARTS, bool VEC, bool FIRST, int LANES>
__global__ void __launch_bounds__((PW + WW) * 32, 1) k_local_state_gather(const ListParams p)
{
    constexpr int kProducerWarps = PW;
    constexpr int kThreads = (PW + WW) * 32;
    constexpr int kBatch = PW * 32 * 4;                       // a batch is four consecutive indices per producer thread
    constexpr int kDepth = 1;                                 // batches a producer thread keeps in flight
    // entry chunks (four steps each) a walker loads before it walks them: seven (items of 5 x 250
    // average 28 steps), four with the 5 + 23 split, whose items average eleven, two for the short
    // items of parts.  Measured: 7 x 500, K = 60, d = 20M: 2.76 ms with 4 or 3, 2.79 with 5;
    // 5 x 250, K = 8, d = 198M: 2.33 ms with 7 or 8, 2.43 with 6, 2.38 with 5
    constexpr int kAhead = PARTS ? 2 : (PW == 5 && WW == 23) ? 4 : 7;
    static_assert(PW + WW <= 32, "the fp64 sums have room for 32 warps");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int vg = (int)blockIdx.x % p.groups, c = (int)blockIdx.x / p.groups;
    const int g = PARTS ? vg % p.wgroups : vg;
    const uint64_t *sched_off = PARTS ? p.sched_off + (size_t)(vg / p.wgroups) * p.part_tiles : p.sched_off;
    const int T = p.T, lm = p.l * p.m;

    const uint32_t smem_base = (uint32_t)__cvta_generic_to_shared(smem_raw);
    int *ctr = reinterpret_cast<int *>(smem_raw);
    unsigned long long *rec_off = reinterpret_cast<unsigned long long *>(smem_raw + 16);
    double *sums = reinterpret_cast<double *>(smem_raw + 64);
    const uint32_t tab_off = kListSmemHead;
    const uint32_t bins_off = tab_off + 2u * (uint32_t)p.tab_bytes;
    const uint32_t ut_off = LANES ? kLaneTiles : bins_off + (uint32_t)lm * 16u;
    const uint32_t ut_bytes = (uint32_t)(T + kListPadRows) * 16u;
    float *bins = reinterpret_cast<float *>(smem_raw + bins_off);
    const uint32_t *prog = LANES ? p.lane_prog + (size_t)(PARTS ? vg / p.wgroups * p.part_tiles : 0) * (p.lane_items + 1) : nullptr;

    if (!LANES)
        for (int t = tid; t < lm * GW; t += kThreads) bins[t] = 0.f;
    for (int t = tid; t < 2 * kListPadRows * GW; t += kThreads) {
        const int b = t / (kListPadRows * GW), r = t % (kListPadRows * GW);
        reinterpret_cast<float *>(smem_raw + ut_off + (size_t)b * ut_bytes)[T * GW + r] = 0.f;
    }
    if (!LANES && tid < 2) ctr[tid] = 0;
    uint4 tab0 = make_uint4(0u, 0u, 0u, 0u);
    if (FIRST) {
        if (!LANES && warp < kProducerWarps) {
            const unsigned long long off = load_u64(sched_off + c);
            if (tid * 16 < p.tab_bytes) tab0 = load_u4(p.sched + off + tid * 16);
            if (tid == 0) rec_off[0] = off;
        }
        fda_grid_wait();
        form_drifts<LINEAR, VEC, 1>(p, g, (int64_t)c * T, warp, PW + WW, smem_base + ut_off, sums + warp * GW * 2);
        __syncthreads();
    } else {
        if (tid < kProducerWarps * GW * 2) sums[tid] = 0.0;
        __syncthreads();
        fda_grid_wait();
    }

    const int n_tiles = p.tiles > c ? (int)((p.tiles - c + p.cpg - 1) / p.cpg) : 0;

    if (warp < kProducerWarps) {
        // =============================== producers ===============================
        const int pt = tid;                                   // quad of indices inside a batch
        // rows of the group; workers past K alias the group's first row (their sums are computed
        // and never written out), so the loop below needs no per-worker predicate
        const float *wbase = p.w + (size_t)(g * GW) * (size_t)p.row_stride;
        int64_t roff[GW];
#pragma unroll
        for (int k = 0; k < GW; ++k) roff[k] = g * GW + k < p.K ? (int64_t)k * p.row_stride : 0;
        float4 wv[kDepth][GW], w0v[kDepth], xv[kDepth];       // four consecutive indices each
        float nf[GW], pf[GW];
#pragma unroll
        for (int k = 0; k < GW; ++k) { nf[k] = 0.f; pf[k] = 0.f; }
        int n_i = FIRST ? 1 : 0, n_c = 0;                 // tile being loaded / stored
        int b_i = 0, b_c = 0;                                 // batch inside it
        uint32_t j_i = (uint32_t)(FIRST ? c + p.cpg : c) * (uint32_t)T + (VEC ? 4 * pt : 128 * warp + lane);   // first index of this thread's next loads
        uint32_t end_i = (uint32_t)((FIRST ? c + p.cpg : c) + 1) * (uint32_t)T;   // end of the tile they belong to
        // 128-index chunks warp, warp + PW, ... of a tile, and the way from behind the last one to the
        // first of this block's next tile
        const int nb = (T / 128 - warp + PW - 1) / PW;
        const uint32_t wrap = (uint32_t)p.cpg * (uint32_t)T - (uint32_t)(nb * kBatch);
        // The rows of a tile two tiles ahead of the one being stored, into L2 (one bulk prefetch per
        // worker row, w_t0 and xi): the producers' loads then find their data in L2.
        auto prefetch_tile = [&](int n) {
            if (n >= n_tiles || pt >= GW + 2) return;
            const int64_t j = (c + n * p.cpg) * (int64_t)T;
            int64_t cnt = p.d - j;
            if (cnt > T) cnt = T;
            uint32_t bytes = (uint32_t)(cnt * 4) & ~15u;
            const float *src = pt < GW ? (g * GW + pt < p.K ? wbase + (int64_t)pt * p.row_stride + j : nullptr)
                                       : (pt == GW ? p.w_t0 + j : (LINEAR ? p.xi + j : nullptr));
            if (!VEC && src) {                                // the 16-byte pieces inside the row
                const uint32_t off = (16u - ((uint32_t)(uintptr_t)src & 15u)) & 15u;
                bytes = (uint32_t)(cnt * 4) > off ? ((uint32_t)(cnt * 4) - off) & ~15u : 0u;
                src += off / 4;
            }
            if (src && bytes)
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
        };
        if (!FIRST) prefetch_tile(0);
        prefetch_tile(1);
        // head of the schedule record of the tile being stored (the walkers' item table) and the
        // record offsets of the next tile, loaded one and two tiles ahead of their use
        uint4 tabv = tab0;
        unsigned long long off0 = 0ull, off1 = 0ull;
        if (!FIRST) {
            off0 = load_u64(sched_off + c);
            off1 = load_u64(sched_off + c + 1);
            if (!LANES && pt * 16 < p.tab_bytes) tabv = load_u4(p.sched + off0 + pt * 16);
            if (!LANES && pt == 0) rec_off[0] = off0;
        }
        if (n_tiles > 1) { off0 = load_u64(sched_off + c + p.cpg); off1 = load_u64(sched_off + c + p.cpg + 1); }
        // the walkers get tile n_c, which is in buffer `buf`
        auto hand_over = [&](int buf) {
            // the table of this tile (loaded a tile ago), the loads of the next one, the offsets
            // of the one after: nothing here waits for memory
            if (!LANES && pt * 16 < p.tab_bytes)
                *reinterpret_cast<uint4 *>(smem_raw + tab_off + (size_t)buf * p.tab_bytes + pt * 16) = tabv;
            if (!LANES && pt == 0) { ctr[buf] = WW; rec_off[(n_c + 1) & 3] = off0; }
            if (n_c + 1 < n_tiles) {
                const unsigned char *nrec = p.sched + off0;
                if (!LANES && pt * 16 < p.tab_bytes) tabv = load_u4(nrec + pt * 16);
                for (uint64_t o = (uint64_t)pt * 128u; o < off1 - off0; o += (uint64_t)kProducerWarps * 32u * 128u)   // the record into L2 ahead of its walk
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(nrec + o));
            }
            if (n_c + 2 < n_tiles) {
                const int64_t t2 = c + (int64_t)(n_c + 2) * p.cpg;
                off0 = load_u64(sched_off + t2);
                off1 = load_u64(sched_off + t2 + 1);
            }
            prefetch_tile(n_c + 2);
            block_barrier<kThreads>();
            b_c = 0;
            ++n_c;
        };
        auto issue = [&](int slot) {
            if (n_i < n_tiles) {
                const float *q = wbase + j_i;
                if (!VEC) {
                    const int64_t left = p.d - (int64_t)j_i;
                    const int n = left > 96 ? 4 : (left > 0 ? (int)(left + 31) / 32 : 0);
#pragma unroll
                    for (int k = 0; k < GW; ++k) wv[slot][k] = load_strided(q + roff[k], n);
                    w0v[slot] = load_strided(p.w_t0 + j_i, n);
                    if (LINEAR) xv[slot] = load_strided(p.xi + j_i, n);
                } else if (end_i <= (uint32_t)p.d) {                    // a whole tile: 128-bit loads
#pragma unroll
                    for (int k = 0; k < GW; ++k) wv[slot][k] = load4_stream(q + roff[k]);
                    w0v[slot] = load4_keep(p.w_t0 + j_i);
                    if (LINEAR) xv[slot] = load4_keep(p.xi + j_i);
                } else {                                      // the last tile of the model
                    const int64_t left = p.d - (int64_t)j_i;
                    const int n = left >= 4 ? 4 : (left > 0 ? (int)left : 0);
#pragma unroll
                    for (int k = 0; k < GW; ++k) wv[slot][k] = load_quad<true>(q + roff[k], n == 4, n);
                    w0v[slot] = load_quad<false>(p.w_t0 + j_i, n == 4, n);
                    if (LINEAR) xv[slot] = load_quad<false>(p.xi + j_i, n == 4, n);
                }
                j_i += kBatch;
                if (++b_i == nb) { b_i = 0; ++n_i; j_i += wrap; end_i += (uint32_t)p.cpg * (uint32_t)T; }
            }
        };
        auto consume = [&](int slot) {
            const int buf = (int)(n_c & 1);
            // rows 4*pt .. 4*pt+3 of the batch; row r is stored at r ^ ((r >> 3) & 3), so that the
            // eight lanes of a store pass hit eight different bank groups (the schedule's entries
            // hold the swizzled row)
            const uint32_t r0 = (uint32_t)(b_c * kBatch) + (VEC ? 4u * pt : fda_list_row(128u * warp + lane));
            const uint32_t dst0 = smem_base + ut_off + (uint32_t)buf * ut_bytes + r0 * 16u;
            const uint32_t sw = (r0 >> 3) & 3u;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float w0 = comp(w0v[slot], q);
                const float u0 = comp(wv[slot][0], q) - w0;
                const float u1 = comp(wv[slot][1], q) - w0;
                const float u2 = comp(wv[slot][2], q) - w0;
                const float u3 = comp(wv[slot][3], q) - w0;
                nf[0] = fmaf(u0, u0, nf[0]); nf[1] = fmaf(u1, u1, nf[1]);
                nf[2] = fmaf(u2, u2, nf[2]); nf[3] = fmaf(u3, u3, nf[3]);
                if (LINEAR) {
                    const float xq = comp(xv[slot], q);
                    pf[0] = fmaf(xq, u0, pf[0]); pf[1] = fmaf(xq, u1, pf[1]);
                    pf[2] = fmaf(xq, u2, pf[2]); pf[3] = fmaf(xq, u3, pf[3]);
                }
                store_row(dst0 + (VEC ? ((uint32_t)q ^ sw) << 4 : 512u * q), u0, u1, u2, u3);
            }
            if (++b_c == nb) {
                // ---- the tile is stored: its item table, its counter, then the hand-over ----
                // (fp32 within the tile: a thread's few indices, then the warp's tree; fp64 across tiles)
                const float a = warp_sums(nf), bq = LINEAR ? warp_sums(pf) : 0.f;
                if ((lane & 7) == 0) {
                    sums[warp * GW * 2 + (lane >> 2)] += (double)a;
                    if (LINEAR) sums[warp * GW * 2 + (lane >> 2) + 1] += (double)bq;
                }
#pragma unroll
                for (int k = 0; k < GW; ++k) { nf[k] = 0.f; pf[k] = 0.f; }
                issue(slot);                                  // (the next loads are on their way across the barrier)
                hand_over(buf);
            } else issue(slot);
        };
#pragma unroll
        for (int s = 0; s < kDepth; ++s) issue(s);
        if (FIRST && n_tiles > 0) hand_over(0);
        while (n_c < n_tiles) {
#pragma unroll
            for (int s = 0; s < kDepth; ++s) {
                if (n_c < n_tiles) consume(s);
            }
        }
    } else if constexpr (LANES > 0) {
        // ===== walkers whose lanes keep their cells: items first, first + WW, .. (`mine` of them) of every tile =====
        const int first = warp - kProducerWarps, mine = max(0, (p.lane_items - first + WW - 1) / WW);
        unsigned long long s01[LANES], s23[LANES];
#pragma unroll
        for (int i = 0; i < LANES; ++i) { s01[i] = 0ull; s23[i] = 0ull; }
        // the program of the warp's next tile: lane i < mine has the word of item i, lane 31 the record's first chunk
        prog += (size_t)c * (p.lane_items + 1) + (lane == 31 ? 0 : 1 + first + lane * WW);
        auto load_prog = [&](int n) {
            return n < n_tiles && (lane < mine || lane == 31) ? __ldg(prog + (size_t)n * p.cpg * (p.lane_items + 1)) : 0u;
        };
        uint32_t next = load_prog(0);
        const uint2 *rec = nullptr, *ent = nullptr;           // of the entries that are asked for
        constexpr int G = kLaneAhead<WW>;
        uint2 nx[G];
        // the next G chunks of an item that has `left` steps left
        auto ask = [&](int left) {
#pragma unroll
            for (int q = 0; q < G; ++q)
                if (left > 4 * q) nx[q] = load_u2(ent + q * kListSlots);
        };
        auto ask_item = [&](uint32_t word) {
            ent = rec + (size_t)(word >> kLaneStepBits) * kListSlots;
            ask((int)(word & ((1u << kLaneStepBits) - 1u)));
        };
        auto ask_tile = [&]() {
            rec = reinterpret_cast<const uint2 *>(p.sched + (size_t)__shfl_sync(0xffffffffu, next, 31) * 256) + lane;
            ask_item(__shfl_sync(0xffffffffu, next, 0));
        };
        ask_tile();
        for (int n = 0; n < n_tiles; ++n) {
            const uint32_t words = next;
            next = load_prog(n + 1);
            block_barrier<kThreads>();                                   // tile n is stored, tile n - 1 is walked
            const uint32_t base = smem_base + ut_off + (uint32_t)(n & 1) * ut_bytes;
            uint32_t word = __shfl_sync(0xffffffffu, words, 0);
#pragma unroll
            for (int i = 0; i < LANES; ++i) {
                if (i >= mine) break;
                const uint32_t then = i + 1 < LANES ? __shfl_sync(0xffffffffu, words, i + 1) : 0u;
                unsigned long long a01 = 0ull, a23 = 0ull;
                for (int left = (int)(word & ((1u << kLaneStepBits) - 1u)); left > 0; left -= 4 * G) {
                    uint2 ch[G];
#pragma unroll
                    for (int q = 0; q < G; ++q) ch[q] = nx[q];
                    if (left > 4 * G) {
                        ent += G * kListSlots;
                        ask(left - 4 * G);
                    } else if (i + 1 < mine) ask_item(then);
                    else ask_tile();
#pragma unroll
                    for (int q = 0; q < G; q += 2) walk_chunks2(ch[q], ch[q + 1], left - 4 * q, base, a01, a23);
                }
                asm("add.rn.f32x2 %0, %0, %1;" : "+l"(s01[i]) : "l"(a01));
                asm("add.rn.f32x2 %0, %0, %1;" : "+l"(s23[i]) : "l"(a23));
                word = then;
            }
        }
        float4 *out = reinterpret_cast<float4 *>(p.part_sk) + (size_t)blockIdx.x * lm;
        // (of the items of a tile those that fill a warp come first)
        const int full = p.m / kListSlots;
        auto row_of = [&](int t) { return t < p.l * full ? t / full : t - p.l * full; };
        auto pos_of = [&](int t) { return (t < p.l * full ? t % full : full) * kListSlots + lane; };
#pragma unroll
        for (int i = 0; i < LANES; ++i) {
            const int row = row_of(first + i * WW), pos = pos_of(first + i * WW);
            if (i >= mine || pos >= p.m) continue;
            const int2 ord = __ldg(p.lane_rows + (PARTS ? vg / p.wgroups * p.l : 0) + row);
            float4 v;
            asm("mov.b64 {%0,%1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(s01[i]));
            asm("mov.b64 {%0,%1}, %2;" : "=f"(v.z), "=f"(v.w) : "l"(s23[i]));
            out[row * p.m + fda_lane_cell(pos, ord.x, ord.y, p.m)] = v;
        }
    } else {
        // =============================== walkers ===============================
        for (int n = 0; n < n_tiles; ++n) {
            block_barrier<kThreads>();                                   // tile n is stored, tile n - 1 is walked
            const int buf = (int)(n & 1);
            // (the record's offset comes from shared memory: a load from L2 here would stand in front of
            // the first entries of every tile)
            const unsigned char *rec = p.sched + rec_off[n & 3];
            const uint32_t *tab = reinterpret_cast<const uint32_t *>(smem_raw + tab_off + (size_t)buf * p.tab_bytes);
            const int n_items = (int)tab[0];
            const uint16_t *cells = reinterpret_cast<const uint16_t *>(rec + fda_sched_cells_off(n_items));
            const unsigned char *ent0 = rec + fda_sched_entries_off(n_items);
            const uint32_t base = smem_base + ut_off + (uint32_t)buf * ut_bytes;
            if constexpr (PARTS) {
                // Short lists (a few steps an item): what an item costs is the way to its entries.  The
                // next item's cell and entries are asked for before this one is walked.
                struct Item { int steps; uint32_t cell; const uint2 *ent; uint2 ch[kAhead]; };
                int it = warp - kProducerWarps;
                auto fetch = [&](Item &x) {
                    const uint32_t d0 = tab[4 + 2 * it], chunk0 = tab[5 + 2 * it];
                    x.steps = (int)(d0 & 0xffffu);
                    x.cell = cells[(size_t)(d0 >> 16) * kListSlots + lane];
                    x.ent = reinterpret_cast<const uint2 *>(ent0 + (size_t)chunk0 * 256) + lane;
#pragma unroll
                    for (int q = 0; q < kAhead; ++q)
                        if (4 * q < x.steps) x.ch[q] = __ldg(x.ent + (size_t)q * kListSlots);
                };
                auto take = [&]() {
                    if (lane == 0) it = atomicAdd(&ctr[buf], 1);
                    it = __shfl_sync(0xffffffffu, it, 0);
                };
                auto walk = [&](Item &x) {
                    unsigned long long a01 = 0ull, a23 = 0ull;
#pragma unroll
                    for (int q = 0; q < kAhead; ++q) walk_chunk(x.ch[q], x.steps - 4 * q, base, a01, a23);
                    for (int c0 = kAhead; 4 * c0 < x.steps; ++c0)
                        walk_chunk(__ldg(x.ent + (size_t)c0 * kListSlots), x.steps - 4 * c0, base, a01, a23);
                    flush_item(bins, lm, x.cell, a01, a23);
                };
                Item a;
                if (it < n_items) fetch(a);
                while (it < n_items) {
                    Item b = a;
                    take();
                    if (it < n_items) fetch(a);
                    walk(b);
                }
            } else {
            int it = warp - kProducerWarps;
            uint32_t d0 = 0, chunk0 = 0;
            if (it < n_items) { d0 = tab[4 + 2 * it]; chunk0 = tab[5 + 2 * it]; }
            while (it < n_items) {
                const int steps = (int)(d0 & 0xffffu);
                const uint32_t cell = cells[(size_t)(d0 >> 16) * kListSlots + lane];
                const uint2 *ent = reinterpret_cast<const uint2 *>(ent0 + (size_t)chunk0 * 256) + lane;
                const int nch = (steps + 3) >> 2;
                if (lane == 0) it = atomicAdd(&ctr[buf], 1);
                it = __shfl_sync(0xffffffffu, it, 0);
                if (it < n_items) { d0 = tab[4 + 2 * it]; chunk0 = tab[5 + 2 * it]; }
                unsigned long long a01 = 0ull, a23 = 0ull;
                // all entry loads of (up to) kAhead chunks first, then the walk: the entries come
                // from global memory (L2), one round trip per kAhead chunks instead of one per chunk
                for (int c0 = 0; c0 < nch; c0 += kAhead) {
                    uint2 ch[kAhead];
#pragma unroll
                    for (int q = 0; q < kAhead; ++q)
                        if (c0 + q < nch) ch[q] = __ldg(ent + (size_t)(c0 + q) * kListSlots);
#pragma unroll
                    for (int q = 0; q + 1 < kAhead; q += 2) walk_chunks2(ch[q], ch[q + 1], steps - 4 * (c0 + q), base, a01, a23);
                    if (kAhead & 1) walk_chunk(ch[kAhead - 1], steps - 4 * (c0 + kAhead - 1), base, a01, a23);
                }
                flush_item(bins, lm, cell, a01, a23);
            }
            }
        }
    }
    block_barrier<kThreads>();                                           // the last tile is walked

    // ---- flush: bins -> this block's partial sketch ----
    if (!LANES) {
        float *out = p.part_sk + (size_t)blockIdx.x * (size_t)lm * GW;
        for (int t = tid; t < lm * GW; t += kThreads) out[t] = bins[t];
    }
    // ---- block partial of (||u||^2, <xi,u>) per worker: the producer warps' sums, in warp order ----
    if (tid < GW * 2) {
        double t = 0.0;
        for (int q = 0; q < (FIRST ? PW + WW : kProducerWarps); ++q) t += sums[q * GW * 2 + tid];
        p.part_np[(size_t)blockIdx.x * GW * 2 + tid] = t;
    }
}

template <int PW, int WW, bool PARTS, bool FIRST, int LANES>
void (*pick_kernel(bool linear, bool vec))(ListParams)
{
    if (linear) return vec ? k_local_state_gather<true, PW, WW, PARTS, true, FIRST, LANES> : k_local_state_gather<true, PW, WW, PARTS, false, FIRST, LANES>;
    return vec ? k_local_state_gather<false, PW, WW, PARTS, true, FIRST, LANES> : k_local_state_gather<false, PW, WW, PARTS, false, FIRST, LANES>;
}

// fda_lanes_*: picks the kernel by the items that a walker warp keeps
template <int PW, int WW, bool PARTS, int LANES>
cudaError_t launch_lanes_n(const ListParams &p, int blocks, bool dependent, cudaStream_t s)
{
    const size_t smem = lane_smem_bytes(p.T);
    auto kern = p.vec ? k_local_state_gather<false, PW, WW, PARTS, true, false, LANES> : k_local_state_gather<false, PW, WW, PARTS, false, false, LANES>;
    if (blocks == 0) return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (dependent) return fda_launch_dependent(kern, blocks, (PW + WW) * 32, smem, s, p);
    kern<<<blocks, (PW + WW) * 32, smem, s>>>(p);
    return cudaGetLastError();
}
template <int PW, int WW, bool PARTS, int MIN, int MAX>
cudaError_t launch_lanes(const ListParams &p, int blocks, bool dependent, cudaStream_t s)
{
    if (p.T % 128 != 0 || p.T < PW * 128 || p.have_xi) return cudaErrorNotSupported;
    if constexpr (MIN == MAX) return p.lane_items <= MAX * WW ? launch_lanes_n<PW, WW, PARTS, MIN>(p, blocks, dependent, s) : cudaErrorNotSupported;
    else return p.lane_items <= MIN * WW ? launch_lanes_n<PW, WW, PARTS, MIN>(p, blocks, dependent, s)
                                          : launch_lanes<PW, WW, PARTS, MIN + 1, MAX>(p, blocks, dependent, s);
}

}  // namespace

#endif
