// List schedule of the sketch kernel (Section 3.1: sk(u)[i][h_i(j)] += s_i(j) u[j]).
//
// The hash of an index depends on (row, index) only, so the order in which a tile's updates
// are applied can be fixed once, when the context is created.  For every tile of T indices
// this file sorts the indices of each sketch row by cell and lays the per-cell lists out as a
// program for the warps of k_local_state_gather:
//
//   * a list holds the indices of one cell (a cell with more than kListMaxLen indices is cut
//     into pieces, flagged so that their sums are added atomically);
//   * a warp walks 32 lists side by side, one per lane: an item.  A lane reads the drift of one
//     index and four workers with one 128-bit shared-memory load per step.  Eight lanes share a
//     pass through shared memory, and the pass is conflict free when their eight rows fall into
//     eight different 16-byte bank groups, i.e. when the indices differ mod 8;
//   * so the lists are grouped by eight (an octet): starting from the longest list left, the
//     builder adds the longest lists whose indices keep every residue class mod 8 of the octet
//     at or below the length of the first one (a class with c indices needs c passes whatever
//     the order), counting a list whose cell shares a bank group with a cell already in the
//     octet (a conflict when the sums are flushed) as two entries shorter.  The entries of an octet are then ordered by decomposing the bipartite
//     multigraph (lists x residue classes, one edge per index, made regular with padding edges)
//     into perfect matchings: in every step each lane reads a different residue class, and a
//     lane with nothing left reads a zero row of a class nobody else reads;
//   * octets are ordered by their number of steps and taken four at a time, items are ordered by
//     steps over all sketch rows of the tile (the kernel hands them out longest first).
//
// Record of one tile (byte offsets; all records are 256-byte aligned, their offsets are in a
// table of tiles + 1 64-bit values):
//   [0]  u32 items   [4] u32 bytes of the record   [8] u32 entry chunks   [12] u32 0
//   [16] items x { u16 steps, u16 cell block, u32 first chunk }, longest first
//   then, 64-byte aligned, cell blocks: [32] u16 cell index i*m + c of the lane's list (bit 15:
//   add atomically; l*m: the lane has no list)
//   then, 256-byte aligned, chunks of 256 bytes: [lane][4] u16 entries, steps 4c .. 4c+3 of an
//   item; entry = row of the drift tile (bits 0..12; index r of the tile is stored in row
//   r ^ ((r >> 3) & 3); T + r is the zero row of class r) | sign << 15.
#include <vector>

#include "fda_hash.cuh"
#include "fda_internal.h"

namespace {

constexpr int kBT = 256;                  // threads of a builder block
constexpr int ML = kListMaxLen;
constexpr int NRES = kListOct;            // residue classes = lanes per shared-memory pass
constexpr int kWindow = 64;               // candidates looked at for every place in an octet
constexpr int kMatchBytes = 288;          // shared memory of the threads that order an octet's entries

struct SchedParams {
    const uint64_t *coeffs;
    int l, m;              // rows of a part, columns
    uint64_t magic;
    int T;
    uint32_t tiles;        // block = part * tiles + tile
    int nl_max;            // lists of a (tile, row)
    int no_max;            // octets of a (tile, row)
    int ni_row_max;        // items of a (tile, row)
    uint32_t *rec_items;   // [tile]  written by the counting pass, read by the writing pass
    uint32_t *rec_chunks;  // [tile]
    uint32_t *rec_steps;   // [tile] steps of all items; all bits set: a cell has more than one list (k_count_lanes)
    const int2 *lane_rows; // order of the cells of every sketch row (of all parts), or null
    uint32_t *lane_prog;   // see fda_ctx (writing pass)
    uint16_t *octets;      // [tile * l + row][9 * no_max] lists and steps of the octets, from the counting pass to the writing pass
    const uint64_t *rec_off;   // [tile + 1] byte offsets of the records (writing pass)
    unsigned char *sched;
};

struct Carve {
    unsigned char *p;
    template <typename T> __device__ T *take(size_t n)
    {
        p = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(p) + 15) & ~(uintptr_t)15);
        T *r = reinterpret_cast<T *>(p);
        p += n * sizeof(T);
        return r;
    }
};

// 16-bit words of the two arrays of hash words, which the matching tables of a row's octets reuse
__host__ __device__ inline size_t hash_words(int T, int ni_row_max)
{
    const size_t tables = (size_t)4 * ni_row_max * kMatchBytes / sizeof(uint16_t);
    return tables > 2 * (size_t)T ? tables : 2 * (size_t)T;
}

// shared memory of a builder block (must match the carve-up in the kernel)
size_t build_smem(int l, int m, int T, int nl_max, int no_max, int ni_row_max)
{
    auto a16 = [](size_t b) { return (b + 15) / 16 * 16; };
    size_t s = 0;
    s += a16(sizeof(int) * m) * 3 + a16(sizeof(int) * (m + 1)) * 2;      // cnt, fill, npiece | start, lfirst
    s += a16(sizeof(uint16_t) * hash_words(T, ni_row_max));               // key, bycell
    s += a16(sizeof(uint16_t) * T);                                       // sorted
    s += a16(sizeof(uint16_t) * nl_max) * 4;                              // ls_start, ls_len, ls_cell, order
    s += a16(8 * (size_t)nl_max);                                         // ls_res
    s += a16(sizeof(int) * (ML + 2)) + a16(sizeof(int) * (kBT + 1));      // cls, scan scratch
    s += a16(sizeof(uint16_t) * 8 * no_max) + a16(sizeof(uint16_t) * no_max) * 2;   // oc_list, oc_cost, oc_order
    s += a16(sizeof(uint32_t) * (size_t)l * ni_row_max) * 3;              // it_steps, it_chunk, it_rank
    s += 64;
    return s + 64;
}

// Exclusive sum of v over the threads of the block; `warps` holds a word per warp and may be used again after the
// next barrier.
__device__ __forceinline__ int block_scan(int v, int *warps)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x / 32;
    int sum = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, sum, off);
        if (lane >= off) sum += o;
    }
    if (lane == 31) warps[warp] = sum;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < warp; ++w) before += warps[w];
    return before + sum - v;
}

// A list that waits for a place in an octet.  info: list number | length << 16 | (cell mod 8) << 23, all bits set
// when there is none; r0, r1: its indices per residue class, a byte each.
struct Cand { uint32_t info, r0, r1; };

// The fullest class of an octet, and the sum of the squares of its classes, when the list comes in
// (cols: two classes to a word; squares: the sum without it)
__device__ __forceinline__ int fullest_with(const uint32_t (&cols)[NRES / 2], const Cand &x)
{
    const uint32_t a = __vmaxu2(cols[0] + __byte_perm(x.r0, 0, 0x4140), cols[1] + __byte_perm(x.r0, 0, 0x4342));
    const uint32_t b = __vmaxu2(cols[2] + __byte_perm(x.r1, 0, 0x4140), cols[3] + __byte_perm(x.r1, 0, 0x4342));
    const uint32_t c = __vmaxu2(a, b);
    return (int)max(c & 0xffffu, c >> 16);
}
__device__ __forceinline__ uint32_t squares_with(const uint32_t (&cols)[NRES / 2], uint32_t squares, const Cand &x)
{
    uint32_t cross = __dp2a_lo(cols[0], x.r0, 0u);
    cross = __dp2a_hi(cols[1], x.r0, cross);
    cross = __dp2a_lo(cols[2], x.r1, cross);
    cross = __dp2a_hi(cols[3], x.r1, cross);
    return __dp4a(x.r1, x.r1, __dp4a(x.r0, x.r0, squares + 2u * cross));
}

// One block per tile (and part of the sketch rows).  WRITE = false: count the items and entry chunks of the record and
// leave the octets for the writing pass; WRITE = true: write the record at its offset.
// Bound: latency (serial chains per octet and per warp), so what counts is how many blocks an SM holds and how many
// threads a chain is shared by: 64 registers and 16-bit hash words for four blocks instead of two, the octets chosen once
// instead of by both passes, eight threads to the matching of an octet instead of one.  fda_create, both
// schedules where there are two: 5 x 250, d = 198M 310 -> 165 ms, d = 7M, K = 30 12.7 -> 8.0; 7 x 500, d = 20M, K = 60 74 -> 36;
// 8 x 1000, d = 2.6M, K = 20 19.0 -> 13.4; 16 x 600, d = 8M 89 -> 45; 5 x 250, d = 61,706 (one schedule) 1.9 -> 1.4.
template <bool WRITE>
__global__ void __launch_bounds__(kBT, 4) k_build_schedule(const SchedParams p)
{
    extern __shared__ __align__(16) unsigned char sm[];
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t rec_no = blockIdx.x;             // records are in order of (part, tile)
    const int64_t tile = blockIdx.x % p.tiles;
    const uint64_t *coeffs = p.coeffs + (size_t)6 * p.l * (blockIdx.x / p.tiles);
    const int T = p.T, m = p.m, NL = p.nl_max, NO = p.no_max;

    Carve cv{sm};
    int *cnt = cv.take<int>(m);
    int *fill = cv.take<int>(m);
    int *npiece = cv.take<int>(m);
    int *start = cv.take<int>(m + 1);
    int *lfirst = cv.take<int>(m + 1);
    uint16_t *key = cv.take<uint16_t>(hash_words(T, p.ni_row_max));   // by index: sign << 15 | cell
    uint16_t *bycell = key + T;                    // the indices grouped by cell
    uint16_t *sorted = cv.take<uint16_t>(T);       // entries (sign << 15 | index), list after list
    uint16_t *ls_start = cv.take<uint16_t>(NL);
    uint16_t *ls_len = cv.take<uint16_t>(NL);
    uint16_t *ls_cell = cv.take<uint16_t>(NL);
    uint16_t *order = cv.take<uint16_t>(NL);       // lists, longest first
    unsigned char *ls_res = cv.take<unsigned char>(8 * (size_t)NL);   // indices per residue class
    int *cls = cv.take<int>(ML + 2);
    int *scan = cv.take<int>(kBT + 1);
    uint16_t *oc_list = cv.take<uint16_t>(8 * (size_t)NO);
    uint16_t *oc_cost = cv.take<uint16_t>(NO);
    uint16_t *oc_order = cv.take<uint16_t>(NO);    // octets, most steps first
    uint32_t *it_steps = cv.take<uint32_t>((size_t)p.l * p.ni_row_max);
    uint32_t *it_chunk = cv.take<uint32_t>((size_t)p.l * p.ni_row_max);
    uint32_t *it_rank = cv.take<uint32_t>((size_t)p.l * p.ni_row_max);
    int *tot = cv.take<int>(8);                    // [0] items so far, [1] chunks so far, [2] lists

    unsigned char *rec = nullptr;
    uint32_t rec_ni = 0;
    size_t cells_off = 0, ent_off = 0;
    if (WRITE) {
        rec = p.sched + p.rec_off[rec_no];
        rec_ni = p.rec_items[rec_no];
        cells_off = fda_sched_cells_off(rec_ni);
        ent_off = fda_sched_entries_off(rec_ni);
    }
    if (tid == 0) { tot[0] = 0; tot[1] = 0; }
    __syncthreads();

    for (int i = 0; i < p.l; ++i) {
        const uint64_t c[6] = {coeffs[6 * i + 0], coeffs[6 * i + 1], coeffs[6 * i + 2],
                               coeffs[6 * i + 3], coeffs[6 * i + 4], coeffs[6 * i + 5]};
        for (int t = tid; t < m; t += kBT) { cnt[t] = 0; fill[t] = 0; }
        if (tid < ML + 2) cls[tid] = 0;
        __syncthreads();

        // ---- hash every index of the tile, count the cells ----
        for (int jl = tid; jl < T; jl += kBT) {
            const uint32_t j = (uint32_t)(tile * T + jl);       // below 2^31 + T
            const uint32_t b = fda::bucket_of(c, j, (uint32_t)m, p.magic);
            const uint32_t sg = fda::sign_is_negative(c, j) ? 0x8000u : 0u;
            key[jl] = (uint16_t)(sg | b);
            atomicAdd(&cnt[b], 1);
        }
        __syncthreads();

        // ---- exclusive scans over the cells: positions and list numbers ----
        const int per = (m + kBT - 1) / kBT;
        {
            int s0 = 0, s1 = 0;
            for (int t = tid * per; t < min(m, (tid + 1) * per); ++t) {
                const int np = (cnt[t] + ML - 1) / ML;
                npiece[t] = np;
                s0 += cnt[t];
                s1 += np;
            }
            int a = block_scan(s0, scan), b = block_scan(s1, scan + kBT / 32);
            for (int t = tid * per; t < min(m, (tid + 1) * per); ++t) {
                start[t] = a; a += cnt[t];
                lfirst[t] = b; b += npiece[t];
            }
            if (tid == kBT - 1) { start[m] = T; lfirst[m] = b; tot[2] = b; }     // (the last thread's b: all lists)
            __syncthreads();
        }
        const int nl = tot[2];

        // ---- group by cell (arrival order), then order every cell's run by index ----
        for (int jl = tid; jl < T; jl += kBT) {
            const int b = key[jl] & 0x7fff;
            bycell[start[b] + atomicAdd(&fill[b], 1)] = (uint16_t)jl;
        }
        __syncthreads();
        for (int pos = tid; pos < T; pos += kBT) {
            const uint32_t idx = bycell[pos], k = key[idx];
            const int b = (int)(k & 0x7fffu);
            int rank = 0;
            for (int q = start[b]; q < start[b + 1]; ++q) rank += bycell[q] < idx ? 1 : 0;
            sorted[start[b] + rank] = (uint16_t)((k & 0x8000u) | fda_list_row(idx));   // the row the index is stored in
        }
        // ---- lists: a cell's run in pieces of nearly equal length ----
        for (int b = tid; b < m; b += kBT) {
            const int n = cnt[b], pieces = npiece[b];
            if (pieces == 0) continue;
            const int base = n / pieces, rem = n % pieces;
            for (int q = 0; q < pieces; ++q) {
                const int it = lfirst[b] + q;
                ls_start[it] = (uint16_t)(start[b] + q * base + min(q, rem));
                ls_len[it] = (uint16_t)(base + (q < rem ? 1 : 0));
                ls_cell[it] = (uint16_t)((i * m + b) | (pieces > 1 ? 0x8000 : 0));
            }
        }
        __syncthreads();
        // ---- inside a list: by residue class, then by index (a stable counting sort) ----
        for (int it = tid; it < nl; it += kBT) {
            uint16_t *e = sorted + ls_start[it];
            const int n = ls_len[it];
            uint16_t tmp[ML];
            int c8[NRES];
#pragma unroll
            for (int r = 0; r < NRES; ++r) c8[r] = 0;
            for (int a = 0; a < n; ++a) { tmp[a] = e[a]; c8[e[a] & (NRES - 1)]++; }
            int pos8[NRES], a0 = 0;
#pragma unroll
            for (int r = 0; r < NRES; ++r) { ls_res[8 * it + r] = (unsigned char)c8[r]; pos8[r] = a0; a0 += c8[r]; }
            for (int a = 0; a < n; ++a) e[pos8[tmp[a] & (NRES - 1)]++] = tmp[a];
            atomicAdd(&cls[n], 1);
        }
        __syncthreads();
        // ---- lists by length, longest first, ties by list number (one warp, 32 lists at a time) ----
        const bool choose = !WRITE && !p.lane_rows;
        if (tid < 32 && choose) {
            int below = 0;                                           // lists that are longer than 64 - 2 * lane
            {
                const int pair = cls[ML - 2 * lane] + cls[ML - 1 - 2 * lane];
                below = pair;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int v = __shfl_up_sync(0xffffffffu, below, off);
                    if (lane >= off) below += v;
                }
                below -= pair;
                const int longer = cls[ML - 2 * lane];
                cls[ML - 2 * lane] = below;
                cls[ML - 1 - 2 * lane] = below + longer;
            }
            __syncwarp();
            for (int it0 = 0; it0 < nl; it0 += 32) {
                const int len = it0 + lane < nl ? (int)ls_len[it0 + lane] : 0;
                const unsigned peers = __match_any_sync(0xffffffffu, len);
                const int at = cls[len] + __popc(peers & ((1u << lane) - 1u));
                __syncwarp();
                if (len > 0) {
                    order[at] = (uint16_t)(it0 + lane);
                    if ((peers >> lane) == 1u) cls[len] = at + 1;       // (the last of them)
                }
                __syncwarp();
            }
        }
        // ---- octets (one warp): the longest list left opens an octet; every further place goes
        // to the longest of the next kWindow lists that keeps all residue classes within the
        // opener's length (ties: a cell whose bank group the octet's flush does not use yet,
        // then the flattest classes); if none fits, to the one that raises the classes least ----
        const int no = p.lane_rows ? (m + NRES - 1) / NRES : (nl + NRES - 1) / NRES;
        if (p.lane_rows) {
            // the octets of the cells' fixed order: 32 neighbours of it are an item in every tile
            const int2 ord = p.lane_rows[(size_t)(blockIdx.x / p.tiles) * p.l + i];
            for (int o = tid; o < no; o += kBT) {
                int cols[NRES], cost = 1;
#pragma unroll
                for (int r = 0; r < NRES; ++r) cols[r] = 0;
                for (int q = 0; q < NRES; ++q) {
                    const int pos = NRES * o + q, cell = pos < m ? fda_lane_cell(pos, ord.x, ord.y, m) : 0;
                    const bool on = pos < m && cnt[cell] > 0;
                    const int li = on ? lfirst[cell] : 0xffff;
                    oc_list[NRES * o + q] = (uint16_t)li;
                    if (!on) continue;
                    cost = max(cost, (int)ls_len[li]);
#pragma unroll
                    for (int r = 0; r < NRES; ++r) cols[r] += ls_res[8 * li + r];
                }
#pragma unroll
                for (int r = 0; r < NRES; ++r) cost = max(cost, cols[r]);
                oc_cost[o] = (uint16_t)cost;
            }
        } else if (!choose) {
            const uint16_t *from = p.octets + (size_t)(rec_no * p.l + i) * 9 * NO;
            for (int x = tid; x < 9 * no; x += kBT) (x < 8 * no ? oc_list[x] : oc_cost[x - 8 * no]) = from[x];
        } else if (tid < 32) {
            // The next kWindow lists that are not placed yet, longest first, in registers: place s of the window
            // in lane s % 32 (lo: the first 32, hi: the others).  A list that is taken leaves the window by moving those
            // behind it up by one; `more` is the list that comes in.
            // Bound: the one warp's chain of some 200 dependent instructions to a place, three quarters of the
            // counting pass, which is why the writing pass reads the octets back.
            auto load = [&](int pos) {
                Cand x{0xffffffffu, 0u, 0u};
                if (pos < nl) {
                    const int li = order[pos];
                    const uint2 r = *reinterpret_cast<const uint2 *>(ls_res + 8 * li);
                    x.info = (uint32_t)li | (uint32_t)ls_len[li] << 16 | (uint32_t)(ls_cell[li] & 7) << 23;
                    x.r0 = r.x; x.r1 = r.y;
                }
                return x;
            };
            Cand lo = load(lane), hi = load(32 + lane), more = load(kWindow);
            int next = kWindow + 1;
            auto from = [&](const Cand &x, int src) {
                return Cand{__shfl_sync(0xffffffffu, x.info, src), __shfl_sync(0xffffffffu, x.r0, src), __shfl_sync(0xffffffffu, x.r1, src)};
            };
            auto take = [&](int w) {
                const Cand got = from(w < 32 ? lo : hi, w & 31);
                const Cand l1 = from(lo, (lane + 1) & 31), h1 = from(hi, (lane + 1) & 31);
                if (lane >= w) lo = lane == 31 ? h1 : l1;
                if (32 + lane >= w) hi = lane == 31 ? more : h1;
                more = load(next++);
                return got;
            };
            for (int o = 0; o < no; ++o) {
                // indices of the octet in the classes 2q, 2q + 1, a half word each, and the sum of their squares
                uint32_t cols[NRES / 2] = {}, squares = 0;
                auto add = [&](const Cand &x) {
                    const uint32_t v[NRES / 2] = {__byte_perm(x.r0, 0, 0x4140), __byte_perm(x.r0, 0, 0x4342),
                                                  __byte_perm(x.r1, 0, 0x4140), __byte_perm(x.r1, 0, 0x4342)};
                    squares = squares_with(cols, squares, x);
#pragma unroll
                    for (int q = 0; q < NRES / 2; ++q) cols[q] += v[q];
                };
                const Cand first = take(0);
                add(first);
                const int L = (int)(first.info >> 16 & 127u);
                unsigned cellmask = 1u << (first.info >> 23);
                if (lane == 0) oc_list[8 * o] = (uint16_t)first.info;
                for (int place = 1; place < NRES; ++place) {
                    uint32_t best = 0xffffffffu;
#pragma unroll
                    for (int half = 0; half < kWindow / 32; ++half) {
                        const Cand &x = half ? hi : lo;
                        const int slot = half * 32 + lane, mx = fullest_with(cols, x), sq = (int)squares_with(cols, squares, x);
                        uint32_t k;
                        if (mx <= L) {
                            const uint32_t conflict = (cellmask >> (x.info >> 23 & 7u)) & 1u;
                            // a flush conflict (two cells of the octet in one bank group) costs about
                            // as much as two idle steps of a lane
                            k = ((uint32_t)(L - (int)(x.info >> 16 & 127u) + 2 * (int)conflict) << 23) |
                                ((uint32_t)min(sq, 0xffff) << 6) | (uint32_t)slot;
                        } else {
                            k = 0x80000000u | ((uint32_t)min(mx, 0x3ff) << 21) |
                                ((uint32_t)min(sq >> 6, 0x7fff) << 6) | (uint32_t)slot;
                        }
                        if (x.info != 0xffffffffu) best = min(best, k);
                    }
                    best = __reduce_min_sync(0xffffffffu, best);
                    if (best == 0xffffffffu) {                       // no list left
                        if (lane == 0) oc_list[8 * o + place] = 0xffffu;
                        continue;
                    }
                    const Cand got = take((int)(best & 63u));
                    add(got);
                    cellmask |= 1u << (got.info >> 23);
                    if (lane == 0) oc_list[8 * o + place] = (uint16_t)got.info;
                }
                if (lane == 0) oc_cost[o] = (uint16_t)max(L, fullest_with(cols, Cand{0u, 0u, 0u}));
            }
        }
        __syncthreads();
        if (choose && p.octets) {
            uint16_t *to = p.octets + (size_t)(rec_no * p.l + i) * 9 * NO;
            for (int x = tid; x < 9 * no; x += kBT) to[x] = x < 8 * no ? oc_list[x] : oc_cost[x - 8 * no];
        }
        // ---- octets by steps (most first, ties by number); four of them make an item ----
        for (int o = tid; o < no; o += kBT) {
            int rank = p.lane_rows ? o : 0;
            const int co = oc_cost[o];
            for (int q = 0; q < no && !p.lane_rows; ++q) rank += (oc_cost[q] > co || (oc_cost[q] == co && q < o)) ? 1 : 0;
            oc_order[rank] = (uint16_t)o;
        }
        __syncthreads();
        const int ni_row = (no + 3) / 4;
        const int item0 = tot[0], chunk0 = tot[1];
        __syncthreads();
        if (tid == 0) {
            int a = chunk0;
            for (int q = 0; q < ni_row; ++q) {
                int steps = oc_cost[oc_order[4 * q]];
                for (int x = 4 * q + 1; p.lane_rows && x < min(no, 4 * q + 4); ++x) steps = max(steps, (int)oc_cost[x]);
                it_steps[item0 + q] = (uint32_t)steps;
                it_chunk[item0 + q] = (uint32_t)a;
                a += (steps + 3) / 4;
            }
            tot[0] = item0 + ni_row;
            tot[1] = a;
        }
        __syncthreads();

        if (WRITE) {
            // ---- cell blocks ----
            uint16_t *cells = reinterpret_cast<uint16_t *>(rec + cells_off);
            for (int t = tid; t < ni_row * kListSlots; t += kBT) {
                const int q = t / kListSlots, ln = t % kListSlots;
                const int pos = 4 * q + ln / NRES;
                uint16_t cell = (uint16_t)(p.l * m);
                if (pos < no) {
                    const int li = oc_list[8 * oc_order[pos] + (ln % NRES)];
                    if (li != 0xffff) cell = ls_cell[li];
                }
                cells[(size_t)(item0 + q) * kListSlots + ln] = cell;
            }
            // ---- entries: a warp per item, eight threads per octet, one to each of its lists ----
            // (with one thread to an octet, four octets to a warp, whose paths differ, an instruction of the
            // matching served one list where it serves up to 32 here)
            uint16_t *ent = reinterpret_cast<uint16_t *>(rec + ent_off);
            for (int q = tid / 32; q < ni_row; q += kBT / 32) {
                const int pos = 4 * q + lane / NRES, s = lane % NRES;
                const int steps = (int)it_steps[item0 + q], padded = (steps + 3) & ~3;
                uint16_t *dst = ent + (size_t)it_chunk[item0 + q] * (kListSlots * 4) + lane * 4;
                // edge[r * 8 + s]: bits 0..6 the indices of list s in class r, bits 7..16 the padding
                // edges that make the graph regular (up to eight full lists in one class: 512), from
                // bit 17 on the list's next entry of the class.  The words live in shared memory (the
                // hash words of the row are no longer needed), what the search itself works on in
                // registers, the same in all eight threads: match (list -> class), back (class -> list), prev
                // and queue, a nibble per entry, 8 for none; alive, a bit per edge, is put together from the threads' rows.
                uint32_t *edge = reinterpret_cast<uint32_t *>(key) + (size_t)pos * (kMatchBytes / 4);
                unsigned short *defL = reinterpret_cast<unsigned short *>(edge + NRES * NRES), *defR = defL + NRES;
                const int o = pos < no ? oc_order[pos] : 0, delta = pos < no ? oc_cost[o] : 0;
                const int li = pos < no ? oc_list[8 * o + s] : 0xffff;
                int a0 = li != 0xffff ? ls_start[li] : 0, len = 0;
                for (int r = 0; r < NRES; ++r) {
                    const int v = li != 0xffff ? ls_res[8 * li + r] : 0;
                    edge[r * NRES + s] = (uint32_t)v | ((uint32_t)a0 << 17);
                    a0 += v;
                    len += v;
                }
                defL[s] = (unsigned short)(delta - len);
                __syncwarp();
                int in_class = 0;
                for (int x = 0; x < NRES; ++x) in_class += (int)(edge[s * NRES + x] & 0x7fu);
                defR[s] = (unsigned short)(delta - in_class);
                __syncwarp();
                if (s == 0)
                    for (int x = 0, r = 0; x < NRES && r < NRES;) {
                        const unsigned dl = defL[x], n = min(dl, (unsigned)defR[r]);
                        edge[r * NRES + x] += n << 7;
                        defL[x] = (unsigned short)(dl - n);
                        defR[r] = (unsigned short)(defR[r] - n);
                        if (dl == n) ++x; else ++r;
                    }
                __syncwarp();
                unsigned row = 0;                                    // the list's edges that exist
                for (int r = 0; r < NRES; ++r) row |= (edge[r * NRES + s] & 0x1ffffu) ? 1u << r : 0u;

                auto nibble = [](unsigned x, int i) { return (int)((x >> (4 * i)) & 15u); };
                auto with = [](unsigned x, int i, int v) { return (x & ~(15u << (4 * i))) | ((unsigned)v << (4 * i)); };
                unsigned match = 0x88888888u;
                unsigned long long word = 0ull;
                for (int t = 0; t < padded; ++t) {
                    // keep the edges of the last matching that still exist, complete it with
                    // augmenting paths (a regular bipartite multigraph has a perfect matching)
                    const int had = nibble(match, s);
                    const bool keep = had < 8 && ((row >> had) & 1u);
                    const unsigned kept = (__ballot_sync(0xffffffffu, keep) >> (lane & 24)) & 0xffu;
                    unsigned back = keep ? (unsigned)(s ^ 8) << (4 * had) : 0u, half = row << (8 * (s & 3));
#pragma unroll
                    for (int x = 1; x < NRES; x <<= 1) back |= __shfl_xor_sync(0xffffffffu, back, x);
                    back ^= 0x88888888u;
                    half |= __shfl_xor_sync(0xffffffffu, half, 1);
                    half |= __shfl_xor_sync(0xffffffffu, half, 2);
                    const unsigned other = __shfl_xor_sync(0xffffffffu, half, 4);
                    const unsigned long long alive = s < 4 ? (unsigned long long)other << 32 | half : (unsigned long long)half << 32 | other;
                    const bool on = t < delta;
                    if (on && kept != 0xffu) {
                        for (int x = 0; x < NRES; ++x)
                            if (!((kept >> x) & 1u)) match = with(match, x, 8);
                        for (int s0 = 0; s0 < NRES; ++s0) {
                            if (nibble(match, s0) < 8) continue;
                            int qh = 0, qt = 1;
                            unsigned vis = 0, prev = 0, queue = (unsigned)s0;
                            bool done = false;
                            while (qh < qt && !done) {
                                const int sq = nibble(queue, qh++);
                                unsigned open = (unsigned)(alive >> (sq * NRES)) & 0xffu & ~vis;
                                vis |= open;
                                for (; open && !done; open &= open - 1u) {
                                    const int r = __ffs((int)open) - 1, owner = nibble(back, r);
                                    prev = with(prev, r, sq);
                                    if (owner < 8) {
                                        queue = with(queue, qt++, owner);
                                        continue;
                                    }
                                    for (int rc = r;;) {
                                        const int sp = nibble(prev, rc), nr = nibble(match, sp);
                                        match = with(match, sp, rc);
                                        back = with(back, rc, sp);
                                        if (sp == s0) break;
                                        rc = nr;
                                    }
                                    done = true;
                                }
                            }
                        }
                    }
                    __syncwarp();
                    uint16_t e = (uint16_t)(T + s);                  // (behind the octet's last step)
                    if (on) {
                        const int r = nibble(match, s) & 7;          // (every list is matched)
                        uint32_t w = edge[r * NRES + s];
                        if (w & 0x7fu) {
                            e = sorted[w >> 17];
                            w += (1u << 17) - 1u;
                        } else {
                            e = (uint16_t)(T + r);
                            w -= 1u << 7;
                        }
                        edge[r * NRES + s] = w;
                        if ((w & 0x1ffffu) == 0u) row &= ~(1u << r);
                    }
                    word |= (unsigned long long)e << (16 * (t & 3));
                    if ((t & 3) == 3) {
                        *reinterpret_cast<unsigned long long *>(dst + (size_t)(t >> 2) * (kListSlots * 4)) = word;
                        word = 0ull;
                    }
                }
            }
        }
        __syncthreads();
    }

    // ---- items of the tile by steps, most first (ties by creation order) ----
    const int ni = tot[0], nch = tot[1];
    for (int q = tid; q < ni; q += kBT) {
        int rank = 0;
        const uint32_t sq = it_steps[q];
        for (int r = 0; r < ni; ++r) rank += (it_steps[r] > sq || (it_steps[r] == sq && r < q)) ? 1 : 0;
        it_rank[q] = (uint32_t)rank;
    }
    __syncthreads();
    if (!WRITE) {
        if (tid == 0) {
            p.rec_items[rec_no] = (uint32_t)ni;
            p.rec_chunks[rec_no] = (uint32_t)nch;
        }
    } else {
        uint32_t *hdr = reinterpret_cast<uint32_t *>(rec);
        if (tid == 0) {
            hdr[0] = (uint32_t)ni;
            hdr[1] = (uint32_t)(ent_off + (size_t)nch * 256);
            hdr[2] = (uint32_t)nch;
            hdr[3] = (ni == (int)rec_ni && nch == (int)p.rec_chunks[rec_no]) ? 0u : 1u;   // 1: the two passes disagree
        }
        for (int q = tid; q < ni; q += kBT) {
            uint32_t *dsc = hdr + 4 + 2 * it_rank[q];
            dsc[0] = (it_steps[q] & 0xffffu) | ((uint32_t)q << 16);
            dsc[1] = it_chunk[q];
            // (in the program the items that fill a warp come first)
            const int per_row = (m + kListSlots - 1) / kListSlots, full = m / kListSlots, of_row = q % per_row;
            const int at = of_row < full ? q / per_row * full + of_row : p.l * full + q / per_row;
            if (p.lane_prog) p.lane_prog[(size_t)rec_no * (ni + 1) + 1 + at] = it_chunk[q] << kLaneStepBits | it_steps[q];
        }
        if (p.lane_prog && tid == 0) p.lane_prog[(size_t)rec_no * (ni + 1)] = (uint32_t)((p.rec_off[rec_no] + ent_off) / 256);
    }
}

// Steps and entry chunks of the items of one tile and sketch row when the row's cells keep the order `ord`: the sums
// over the items that this thread looks at.  cls8: m * 8 words of shared memory.  `bad` is set when a cell
// has more than one list.  (k_build_schedule comes to the same numbers by sorting; only counting is done here.)
__device__ void count_lane_items(const uint64_t *c, int2 ord, int m, uint64_t magic, int T, uint32_t tile, int *cls8,
                                 uint32_t &steps, uint32_t &chunks, uint32_t &bad)
{
    const int tid = threadIdx.x;
    for (int t = tid; t < 8 * m; t += kBT) cls8[t] = 0;
    __syncthreads();
    for (int r = tid; r < T; r += kBT)
        atomicAdd(&cls8[8 * fda::bucket_of(c, tile * (uint32_t)T + r, (uint32_t)m, magic) + (fda_list_row(r) & 7)], 1);
    __syncthreads();
    for (int q = tid; q < (m + 31) / 32; q += kBT) {
        int most = 1;
        for (int o = 0; o < 4; ++o) {
            int cols[8] = {};
            for (int x = 0; x < 8; ++x) {
                const int pos = 32 * q + 8 * o + x;
                if (pos >= m) break;
                const int *v = cls8 + 8 * fda_lane_cell(pos, ord.x, ord.y, m);
                int len = 0;
                for (int k = 0; k < 8; ++k) { len += v[k]; cols[k] += v[k]; }
                most = max(most, len);
                if (len > ML) bad = 1;
            }
            for (int k = 0; k < 8; ++k) most = max(most, cols[k]);
        }
        steps += most;
        chunks += (most + 3) / 4;
    }
    __syncthreads();
}

// Score of an order of a sketch row's cells for lanes that keep their cells: steps of its items over
// kSamples tiles.  Block (shift, row) looks at the order in which index j + e lies in the cell after that of
// j, for e = 2 * shift + 1, unless the bucket hash wraps around p between the two: bucket(j + e) - bucket(j) is
// r mod m, r = a * e mod p, except for a share |r| / p of all j.  The lists of eight neighbours of that
// order are then copies of one another, shifted by e, 2e, ..: as long as one another, and - e being odd - spread
// over the residue classes.  Scores of cells that need several lists: all bits set.
constexpr int kShifts = 256, kSamples = 3;

__device__ int2 cell_order(uint64_t a, uint32_t e, int m)
{
    uint64_t r = fda::mul_add_mod_p(a, e, 0);
    int step = (int)(r % (uint64_t)m);
    if (r > fda::kP61 / 2) {                       // r - p is the nearer one
        step = (int)((fda::kP61 - r) % (uint64_t)m);
        step = step ? m - step : 0;
    }
    int x = m, y = step;
    while (y) { const int t = x % y; x = y; y = t; }
    return make_int2(step, m / x);
}

__global__ void __launch_bounds__(kBT) k_score_orders(const uint64_t *coeffs, int m, uint64_t magic, int T, uint32_t tiles, uint32_t *score)
{
    extern __shared__ int cls8[];                  // [m][8] indices of a cell by residue class
    __shared__ uint32_t sum[kBT / 32];
    const uint64_t *c = coeffs + 6 * blockIdx.y;
    const uint32_t e = 2 * blockIdx.x + 1;
    const int tid = threadIdx.x;
    const int2 ord = cell_order(c[0], e, m);
    const bool same = ord.x == 0 && m > 1;         // j and j + e share a cell: no order
    uint32_t steps = 0, chunks = 0, bad = same;
    for (int smp = 0; smp < kSamples && !same; ++smp)
        count_lane_items(c, ord, m, magic, T, (uint32_t)((uint64_t)(tiles - 1) * smp / (kSamples - 1)), cls8, steps, chunks, bad);
    steps = __reduce_add_sync(0xffffffffu, steps);
    bad = __any_sync(0xffffffffu, bad);
    if ((tid & 31) == 0) sum[tid / 32] = bad ? 0xffffffffu : steps;
    __syncthreads();
    if (tid == 0) {
        uint32_t t = 0;
        for (int w = 0; w < kBT / 32; ++w) t = sum[w] == 0xffffffffu || t == 0xffffffffu ? 0xffffffffu : t + sum[w];
        score[blockIdx.y * kShifts + blockIdx.x] = t;
    }
}

// Counting pass of the schedule whose cells stay with their lanes: a block per record.
__global__ void __launch_bounds__(kBT) k_count_lanes(const SchedParams p)
{
    extern __shared__ int cls8[];
    __shared__ uint32_t sum[3];
    const uint32_t part = blockIdx.x / p.tiles, tile = blockIdx.x % p.tiles;
    uint32_t steps = 0, chunks = 0, bad = 0;
    if (threadIdx.x < 3) sum[threadIdx.x] = 0;
    for (int i = 0; i < p.l; ++i)
        count_lane_items(p.coeffs + 6 * (part * p.l + i), p.lane_rows[part * p.l + i], p.m, p.magic, p.T, tile, cls8, steps, chunks, bad);
    steps = __reduce_add_sync(0xffffffffu, steps);
    chunks = __reduce_add_sync(0xffffffffu, chunks);
    bad = __reduce_or_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0) { atomicAdd(&sum[0], steps); atomicAdd(&sum[1], chunks); atomicOr(&sum[2], bad); }
    __syncthreads();
    if (threadIdx.x == 0) {
        p.rec_items[blockIdx.x] = (uint32_t)(p.l * ((p.m + kListSlots - 1) / kListSlots));
        p.rec_chunks[blockIdx.x] = sum[1];
        p.rec_steps[blockIdx.x] = sum[2] ? 0xffffffffu : sum[0];
    }
}

// the best order of every row (a warp each)
__global__ void k_pick_orders(const uint64_t *coeffs, int m, const uint32_t *score, int2 *rows)
{
    const int row = blockIdx.x, lane = threadIdx.x;
    uint32_t best = 0xffffffffu, at = 0;
    for (int i = lane; i < kShifts; i += 32)
        if (score[row * kShifts + i] < best) { best = score[row * kShifts + i]; at = i; }
    const uint32_t least = __reduce_min_sync(0xffffffffu, best);
    at = __reduce_min_sync(0xffffffffu, best == least ? at : 0xffffu);
    if (lane == 0) rows[row] = least == 0xffffffffu ? make_int2(1, m) : cell_order(coeffs[6 * row], 2 * at + 1, m);
}

}  // namespace

// The largest tile (a multiple of kListBatch indices) whose two drift buffers fit beside the bins of
// `rows` sketch rows, or 0 when its lists would be shorter than min_len entries on average: short lists
// do not pay for their flushes.
static int list_tile_indices(const fda_ctx *ctx, int rows, int min_len, int *ni_max_out)
{
    const int m = ctx->m;
    if (rows * m + 1 >= 0x8000) return 0;
    for (int T = kListMaxTile; T >= 2 * kListBatch; T -= kListBatch) {
        const int nl = (m < T ? m : T) + T / kListMaxLen;
        const int ni_max = rows * ((nl + kListSlots - 1) / kListSlots);
        if (fda_list_smem_bytes(rows, m, T, ni_max) > (size_t)ctx->smem_optin) continue;
        if (T < min_len * m) return 0;
        *ni_max_out = ni_max;
        return T;
    }
    return 0;
}

// Walker warps for a block's `items` items of `rows` sketch rows (every other warp of 28 to 32 produces).
// Up to three rows the producers set the pace: no more than 20 walkers beside 12 of them.  Measured, K = 8, d = 20M, us with
// 12 / 16 / 20 / 23 / 24 walkers: 3 x 250 (24 items) 158 / 156 / 185 / 204 / 214; 2 x 320 (20) 142 / 142 / 156 / 197 / 197; 3 x 320 (30)
// 179 / 160 / 164 / 201 / 207; 3 x 500 (48) 187 / 177 / 173 / 207 / 211; 2 x 1000 (64) 203 / 183 / 168 / 199 / 197; 3 x 800 (75) 248 / 216 /
// 187 / 211 / 209.  From four rows on the walk does: one item to a warp where 12, 16 or 20 warps have that, two up to
// 32 items, beyond that as many warps as leave the fewest lanes without a cell, and of those that leave equally
// many the fewest; from 61 items on 20 are too few.  4 x 100 (16 items) 246 / 203 / 209 / 224 / 226; 8 x 64 (16) 373 / 289 / 310 / 299 / 296;
// 5 x 128 (20) 221 / 239 / 199 / 230 / 231; 8 x 96 (24) 279 / 287 / 373 / 361 / 277; 5 x 160 (25) 244 / 205 / 258 / 249 / 245; 5 x 250 (40) 241 /
// 232 / 207 / 224 / 229; 6 x 200 (42) 287 / 278 / 300 / 244 / 252; 6 x 250 (48) 254 / 252 / 279 / 275 / 246; 7 x 250 (56) 309 / 310 / 283 /
// 286 / 297; 5 x 400 (65) 330 / 306 / 273 / 231 / 234; 5 x 500 (80) 299 / 262 / 240 / 227 / 229; 6 x 500 (96) - / 321 / 285 / 273 / 256;
// 7 x 500 (112) - / 366 / 322 / 290 / 310; 8 x 500 (128) - / - / 394 / 354 / 362.  It misses by up to 6 % at 4 x 350 (44 items, 216 with 23,
// 205 with 16) and 2 x 640 (40, 168 with 20, 158 with 16).
static int lane_walkers(int rows, int items)
{
    if (rows > 3)
        for (int w : {12, 16, 20})
            if (items <= w) return w;
    if (items <= 24) return 12;
    if (items <= 32) return 16;
    if (rows <= 3) return 20;
    int best = items <= 60 ? 20 : 23;
    for (int w : {23, 24})
        if ((items + w - 1) / w * w < (items + best - 1) / best * best) best = w;
    return best;
}

// Geometry of the schedule when cells stay with their lanes: there are no bins, so the tile depends on the lists only.
// Six batches of 1024 indices, fewer where lists would come near their limit, seven where they would be
// shorter than ten entries (5 x 250, K = 8, d = 198M: 1860 us with six, 1907 with seven, 1991 with five; 8 x 1000,
// K = 20, d = 2.6M: 165 with seven, 189 with six).  The sketch rows go in one part unless their items would
// be more than a block's lanes can keep.
static int lane_geometry(const fda_ctx *ctx, int *parts_out, int *ni_max_out)
{
    const int m = ctx->m;
    int T = 6 * kListBatch;
    if (T < 10 * m) T += kListBatch;
    while (T > 56 * m && T > 2 * kListBatch) T -= kListBatch;
    if (T < 5 * m || T > 56 * m) return 0;
    // Where a quarter of the lanes would have no cell, or lists that come near their limit leave tiles of two batches, the list
    // kernel is as fast or faster up to twelve rows.  Measured, K = 8, d = 20M, us, list kernel and this one: of the 96 lanes of
    // 65 columns 31 idle, 3 x 65 212 and 219, 5 x 65 331 and 350, 8 x 65 387 and 398; 12 x 70 558 and 567; tiles of two batches:
    // 3 x 48 212 and 231, 8 x 50 420 and 458, 5 x 50 281 and 275; but 16 x 65 777 and 660, 16 x 44 779 and 699.  On the other side of
    // the line 3 x 72 208 and 206, 8 x 72 373 and 354, 8 x 97 391 and 325, 8 x 100 387 and 328, 3 x 100 206 and 177,
    // 5 x 56 275 and 238, 8 x 56 400 and 379.
    if (m < 128 && ctx->l <= 12 && ((m + kListSlots - 1) / kListSlots * kListSlots * 3 > 4 * m || T < 3 * kListBatch)) return 0;
    for (int parts = 1; parts <= 4; parts *= 2) {
        if (ctx->l % parts) break;
        const int rows = ctx->l / parts, items = rows * ((m + kListSlots - 1) / kListSlots);
        if (items > kLaneMaxItems || rows * m + 1 >= 0x8000) continue;
        const int groups = (ctx->K_max + kListWorkers - 1) / kListWorkers * parts;
        if (!fda_lanes_pay((ctx->d_max + T - 1) / T, groups, ctx->n_sm)) return 0;
        *parts_out = parts;
        *ni_max_out = items;
        return T;
    }
    return 0;
}

// Geometry of the schedule: all rows in one part where lists of six entries fit, else two or four
// equal parts of the rows, each with bins, records and blocks of its own, from five entries on: a part
// forms the drifts again (its loads hit L2), but the bins it does not hold make room for lists twice as
// long.  8 x 1000 as two parts of 4 x 1000: tiles of 5120 indices instead of 3072.
static int list_geometry(const fda_ctx *ctx, int *parts_out, int *ni_max_out)
{
    if (ctx->l == 0) return 0;
    for (int parts = 1; parts <= 4; parts *= 2) {
        if (ctx->l % parts) break;
        const int T = list_tile_indices(ctx, ctx->l / parts, parts == 1 ? 6 : 5, ni_max_out);
        if (T) { *parts_out = parts; return T; }
    }
    return 0;
}

// What the writing pass of a schedule still reads when build_schedule has returned (bytes: also what was
// pending before, which counts as free memory).
struct PendingBuild {
    uint32_t *items = nullptr;
    size_t bytes = 0;
};

// Builds one of the two schedules on stream s; none is built (and cudaSuccess returned) for a sketch, a hash, a size or a
// memory limit that it does not suit.  The writing pass is left running.
static cudaError_t build_schedule(fda_ctx *ctx, bool lanes, cudaStream_t s, PendingBuild &pending)
{
    int ni_max = 0, parts = 1;
    const int T = lanes ? lane_geometry(ctx, &parts, &ni_max) : list_geometry(ctx, &parts, &ni_max);
    if (T == 0) return cudaSuccess;
    const int64_t part_tiles = (ctx->d_max + T - 1) / T, tiles = part_tiles * parts;      // records
    if (tiles > 0x7fffffffLL) return cudaSuccess;

    SchedParams p{};
    p.coeffs = ctx->coeffs_dev; p.l = ctx->l / parts; p.tiles = (uint32_t)part_tiles; p.m = ctx->m; p.magic = ~0ull / (uint64_t)ctx->m;
    p.T = T;
    p.nl_max = (ctx->m < T ? ctx->m : T) + T / kListMaxLen;
    p.no_max = (p.nl_max + kListOct - 1) / kListOct;
    p.ni_row_max = (p.nl_max + kListSlots - 1) / kListSlots;
    const size_t bsmem = build_smem(p.l, p.m, T, p.nl_max, p.no_max, p.ni_row_max);
    if (bsmem > (size_t)ctx->smem_optin) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_build_schedule<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bsmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_build_schedule<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bsmem);
    if (e != cudaSuccess) return e;

    uint32_t *items = nullptr, *chunks = nullptr, *steps = nullptr, *score = nullptr;
    int2 *rows = nullptr;
    uint32_t *prog = nullptr;
    uint64_t *off = nullptr;
    unsigned char *buf = nullptr;
    auto cleanup = [&]() { cudaFree(items); cudaFree(rows); cudaFree(prog); cudaFree(off); cudaFree(buf); };
    // one allocation for what only the builder needs (the octets take a twentieth to a fifth of what the schedule does, so without
    // room for them there is none for the schedule: then it is only counted)
    const size_t words = 3 * (size_t)tiles + (size_t)ctx->l * kShifts, octet_bytes = lanes ? 0 : sizeof(uint16_t) * 9 * (size_t)tiles * p.l * p.no_max;
    if (octet_bytes && cudaMalloc(&items, sizeof(uint32_t) * words + octet_bytes) == cudaSuccess) p.octets = reinterpret_cast<uint16_t *>(items + words);
    else cudaGetLastError();
    if ((!items && cudaMalloc(&items, sizeof(uint32_t) * words) != cudaSuccess) ||
        (lanes && cudaMalloc(&rows, sizeof(int2) * ctx->l) != cudaSuccess) ||
        cudaMalloc(&off, sizeof(uint64_t) * (tiles + 1)) != cudaSuccess) {
        cudaGetLastError();
        cleanup();
        return cudaSuccess;
    }
    chunks = items + tiles; steps = chunks + tiles; score = steps + tiles;
    p.rec_items = items; p.rec_chunks = chunks; p.rec_steps = steps;
    std::vector<uint32_t> h_count(3 * (size_t)tiles);
    const uint32_t *h_items = h_count.data(), *h_chunks = h_items + tiles, *h_steps = h_chunks + tiles;
    std::vector<uint64_t> h_off((size_t)tiles + 1);
    auto count = [&]() {
        if (lanes) k_count_lanes<<<(unsigned)tiles, kBT, sizeof(int) * 8 * (size_t)ctx->m, s>>>(p);
        else k_build_schedule<false><<<(unsigned)tiles, kBT, bsmem, s>>>(p);
        cudaError_t r = cudaGetLastError();
        if (r == cudaSuccess) r = cudaMemcpyAsync(h_count.data(), items, sizeof(uint32_t) * 3 * tiles, cudaMemcpyDeviceToHost, s);
        return r == cudaSuccess ? cudaStreamSynchronize(s) : r;
    };
    if (lanes) {
        const size_t score_smem = sizeof(int) * 8 * (size_t)ctx->m;
        if (score_smem > 48 * 1024) { cleanup(); return cudaSuccess; }
        k_score_orders<<<dim3(kShifts, (unsigned)ctx->l), kBT, score_smem, s>>>(ctx->coeffs_dev, ctx->m, p.magic, T, p.tiles, score);
        k_pick_orders<<<(unsigned)ctx->l, 32, 0, s>>>(ctx->coeffs_dev, ctx->m, score, rows);
        p.lane_rows = rows;
    }
    e = count();
    if (e == cudaSuccess && lanes) {
        uint64_t total_steps = 0;
        bool fits = true;
        for (int64_t t = 0; t < tiles; ++t) { fits = fits && h_steps[t] != 0xffffffffu; total_steps += h_steps[t]; }
        // (even hashes need 1.1 to 1.35 steps per entry, one uneven row of five or seven puts the sum far above 1.6)
        if (!fits || total_steps * kListSlots * 10 > (uint64_t)16 * tiles * p.l * T) { cleanup(); return cudaSuccess; }
    }
    if (e != cudaSuccess) { cleanup(); return e; }
    uint64_t total = 0;
    for (int64_t t = 0; t < tiles; ++t) {
        h_off[t] = total;
        if ((int)h_items[t] > ni_max) { cleanup(); return cudaSuccess; }      // cannot happen; stay with the other kernels
        total += fda_sched_entries_off(h_items[t]) + (uint64_t)h_chunks[t] * 256;
    }
    h_off[tiles] = total;
    const int lane_items = p.l * ((ctx->m + kListSlots - 1) / kListSlots);
    const uint64_t prog_bytes = lanes ? sizeof(uint32_t) * (uint64_t)(lane_items + 1) * tiles : 0;
    const uint64_t all_bytes = total + prog_bytes + ctx->sched_bytes;         // (of both schedules, when this is the second)
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess || (!lanes && !p.octets) || total + prog_bytes > (free_b + octet_bytes + pending.bytes) / 3 ||
        (ctx->sched_limit_bytes > 0 && all_bytes > (uint64_t)ctx->sched_limit_bytes) ||
        cudaMalloc(&buf, total) != cudaSuccess || (lanes && cudaMalloc(&prog, prog_bytes) != cudaSuccess)) {
        cudaGetLastError();
        cleanup();
        (lanes ? ctx->lane_skipped_bytes : ctx->sched_skipped_bytes) = total + prog_bytes;
        return cudaSuccess;                                                   // leave the memory to the models
    }
    e = cudaMemcpyAsync(off, h_off.data(), sizeof(uint64_t) * (tiles + 1), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) { cleanup(); return e; }
    p.rec_off = off; p.sched = buf;
    p.lane_prog = prog;
    k_build_schedule<true><<<(unsigned)tiles, kBT, bsmem, s>>>(p);
    e = cudaGetLastError();
    if (e != cudaSuccess) { cudaDeviceSynchronize(); cleanup(); return e; }
    pending.items = items; pending.bytes = sizeof(uint32_t) * words + octet_bytes;
    if (lanes) {
        ctx->lane_sched = buf; ctx->lane_off = off; ctx->lane_prog = prog; ctx->lane_rows = rows;
        ctx->lane_records = total;
        ctx->lane_bytes = total + prog_bytes + sizeof(uint64_t) * (tiles + 1) + sizeof(int2) * ctx->l;
        ctx->lane_T = T; ctx->lane_parts = parts; ctx->lane_tiles = part_tiles;
        ctx->lane_items = lane_items; ctx->lane_walkers = lane_walkers(p.l, lane_items);
        return cudaSuccess;
    }
    ctx->sched = buf; ctx->sched_off = off; ctx->sched_bytes = total; ctx->sched_T = T;
    ctx->sched_ni_max = ni_max; ctx->sched_tiles = part_tiles; ctx->sched_parts = parts;
    return cudaSuccess;
}

// The second schedule is begun while the first one's writing pass runs: on short vectors, which fill few SMs, both are
// bound by latency.  fda_create, one after the other and so: 5 x 250, K = 14, d = 1.2M 4.2 and 3.5 ms, 7 x 500, K = 44, d = 0.6M 5.6 and 4.8,
// 5 x 250, K = 30, d = 7M 8.8 and 8.5, 8 x 1000, K = 20, d = 2.6M 14.3 and 13.9.
cudaError_t fda_build_schedules(fda_ctx *ctx, bool second)
{
    PendingBuild first, last;
    cudaError_t e = build_schedule(ctx, false, nullptr, first);
    last.bytes = first.bytes;
    if (e == cudaSuccess && ctx->sched && second) e = build_schedule(ctx, true, ctx->side_stream, last);
    const cudaError_t done = cudaDeviceSynchronize();
    cudaFree(first.items);
    cudaFree(last.items);
    return e != cudaSuccess ? e : done;
}
