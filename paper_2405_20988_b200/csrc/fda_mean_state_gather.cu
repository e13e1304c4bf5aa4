// Averaged state on the list schedule (fda_mean_state on a context that holds one).
//
// By the linearity of the sketch (Section 3.1, property (a)) the sketch of the mean drift
// u-bar = (1/K) sum_k u^(k) is the average of the K worker sketches, so the cells of S-bar cost l
// updates per index instead of K*l.  This kernel is the sibling of k_local_state_gather
// (fda_local_state_gather.cu) and walks the same schedule (fda_sched.cu): a block serves all K
// workers and a strided set of tiles, producers fill a tile in shared memory, walkers gather from
// it, one block-wide barrier per tile hands the two tile buffers over.  What differs:
//
//   * a row of the tile is one float - the sum over the workers of the drifts of the index - and a
//     cell of the bins one float, so a walker does a 32-bit shared-memory load per entry (the
//     schedule keeps the eight lanes of an octet in different banks mod 8; lanes of different
//     octets may still share a bank) and keeps one sum; everything is divided by K at the end;
//   * the single-column tile leaves most of the shared memory free, and the loads land there
//     instead of in registers: the rows of a quad of indices (the K workers, w_t0, xi) are copied
//     asynchronously, `depth` slots ahead per thread, and read back when their group has landed
//     (cp.async.wait_group: nothing here can wait for ever).  A slot holds the quad of up to ten
//     rows; more workers arrive in several slots, so that the bytes in flight depend on neither
//     registers, the number of producer warps nor K.  Rows that are not 16-byte aligned, and the end
//     of the model, are copied four bytes at a time, 32 consecutive indices per warp instruction,
//     with zeros for what lies past the end;
//   * 8 producer and 24 walker warps at 64 registers.
//
// Measured on B200, 5 x 250, K = 8, d = 198M, one pass: 1.50 ms (0.73 of
// the measured copy bandwidth).  On the way: loads landing in registers four rows at a time with
// a four-column tile and 12 + 16 warps 2.15 ms; single-column tile 2.07; landing zone with 8 + 20
// warps 1.73, with 8 + 24 warps 1.67 (6 + 26: 1.86; 12 + 16: 2.01; 4 + 24: 2.12; depth capped at
// 3 / 2: 1.76 / 1.95); without the L2 prefetch of the next tiles' rows that the per-worker kernel
// issues, 1.56; with every shared-memory region on a 128-byte boundary, 1.50.  7 x 500, K = 60,
// d = 20M, where the drifts used to be averaged in a pass of their own first: 0.93 -> 0.82 ms.
//
// k_mean_sketch_short, below, walks the same schedule over the single row of averaged drifts that k_mean_model has
// left in device memory (the two scalars are then that kernel's).

#include <algorithm>

#include "fda_internal.h"
#include "fda_list_kernel.cuh"

namespace {

using namespace fda_list;

constexpr int kPW = 8;                         // producer warps
constexpr int kBatch = kPW * 32 * 4;           // a batch is four consecutive indices per producer thread
constexpr int kWW = 24;                        // walker warps
constexpr int kThreads = (kPW + kWW) * 32;
constexpr uint32_t kRowPitch = kPW * 32u * 16u;   // one row of a landing-zone slot: 16 bytes per producer thread
constexpr int kMaxDepth = 8;
constexpr int kMaxPiece = 10;                  // rows of a landing-zone slot

struct MeanParams {
    ListParams q;                    // rows, schedule, partial-sum buffers
    int piece;                       // rows of a landing-zone slot: a quad of K rows arrives in K / piece slots
    int depth;                       // slots a producer thread keeps in flight (1 .. kMaxDepth)
};

// 16 bytes from global memory straight into shared memory (no register in between), in groups
// that the issuing thread waits for by age.
__device__ __forceinline__ void cp_async16(uint32_t dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// four bytes (on == false: four zero bytes, src is not read)
__device__ __forceinline__ void cp_async4(uint32_t dst, const float *src, bool on)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(on ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// returns when at most n (0..7) of the thread's groups are still in flight
__device__ __forceinline__ void cp_async_wait_upto(int n)
{
    switch (n) {
        case 0: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
        case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
        case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
        case 3: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
        case 4: asm volatile("cp.async.wait_group 4;" ::: "memory"); break;
        case 5: asm volatile("cp.async.wait_group 5;" ::: "memory"); break;
        case 6: asm volatile("cp.async.wait_group 6;" ::: "memory"); break;
        default: asm volatile("cp.async.wait_group 7;" ::: "memory"); break;
    }
}
__device__ __forceinline__ float4 lds128(uint32_t addr)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
// One entry: a 32-bit load of the row, the entry's sign flips the top bit.
__device__ __forceinline__ void gather1(uint32_t e, uint32_t base, float &a)
{
    float u;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(u) : "r"(base + ((e & 0x1fffu) << 2)));
    a += __uint_as_float(__float_as_uint(u) ^ ((e & 0x8000u) << 16));
}

// one chunk of an item: the steps that are left of it, at most four
__device__ __forceinline__ void gather1_chunk(const uint2 &ch, int left, uint32_t base, float &a)
{
    if (left >= 4) {
        gather1(ch.x & 0xffffu, base, a);
        gather1(ch.x >> 16, base, a);
        gather1(ch.y & 0xffffu, base, a);
        gather1(ch.y >> 16, base, a);
    } else if (left > 0) {
        gather1(ch.x & 0xffffu, base, a);
        if (left > 1) gather1(ch.x >> 16, base, a);
        if (left > 2) gather1(ch.y & 0xffffu, base, a);
    }
}
// the sum of a lane's list into the bins
__device__ __forceinline__ void flush1(float *bins, int lm, uint32_t cell, float a)
{
    if ((cell & 0x7fffu) < (uint32_t)lm) {
        float *b = bins + (cell & 0x7fffu);
        if (cell & 0x8000u) atomicAdd(b, a);                // a cell with several lists
        else *b += a;
    }
}

// Shared-memory offsets: every region starts on a 128-byte boundary (the 16-byte stores and the
// asynchronous copies need 16; with the landing zone 48 bytes off a 128-byte boundary the pass ran
// 8 % slower).
__host__ __device__ inline uint32_t align128(uint32_t b) { return (b + 127u) & ~127u; }
__host__ __device__ inline uint32_t mean_bins_off(int tab_bytes) { return align128(kListSmemHead + 2u * (uint32_t)tab_bytes); }
__host__ __device__ inline uint32_t mean_ut_off(int lm, int tab_bytes) { return align128(mean_bins_off(tab_bytes) + (uint32_t)lm * 4u); }
__host__ __device__ inline uint32_t mean_ut_bytes(int T) { return align128((uint32_t)(T + kListPadRows) * 4u); }
// bytes in front of the landing zone: counters and sums, two item tables, bins, two tile buffers
inline size_t mean_smem_fixed(int l, int m, int T, int tab_bytes)
{
    return (size_t)mean_ut_off(l * m, tab_bytes) + 2 * (size_t)mean_ut_bytes(T);
}

// Shared-memory plan (bytes from the start of dynamic shared memory):
//   [0, 8)      item counters of the two tile buffers
//   [16, 48)    offsets of the schedule records of the tiles n, n + 1 (slot n mod 4)
//   [64, 192)   sums[producer warp][2] (fp64): sum_k ||u_k||^2 and <xi, sum_k u_k> over the tiles so far
//   [2112, ..)  two item tables (tab_bytes each): the head of a tile's schedule record
//   then        bins[l*m]
//   then        ut[2][T + 8]   (summed drifts; eight zero rows behind each)
//   then        the landing zone: depth slots of R rows of kRowPitch bytes
// (each region on a 128-byte boundary)
// AHEAD: entry chunks (four steps each) a walker loads before it walks them: eight, or five for the short
// items of sketches of seven or more rows (k_local_state_gather has a rule of its own).
// MULTI: the rows of a quad arrive in several slots (more than kMaxPiece rows).
// VEC: w, w_t0 and xi are 16-byte aligned.
template <bool LINEAR, int AHEAD, bool MULTI, bool VEC>
__global__ void __launch_bounds__(kThreads, 1) k_mean_state_gather(const MeanParams mp)
{
    const ListParams &p = mp.q;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c = (int)blockIdx.x;
    const int T = p.T, lm = p.l * p.m;

    const uint32_t smem_base = (uint32_t)__cvta_generic_to_shared(smem_raw);
    int *ctr = reinterpret_cast<int *>(smem_raw);
    unsigned long long *rec_off = reinterpret_cast<unsigned long long *>(smem_raw + 16);
    double *sums = reinterpret_cast<double *>(smem_raw + 64);
    const uint32_t tab_off = kListSmemHead;
    const uint32_t bins_off = mean_bins_off(p.tab_bytes);
    const uint32_t ut_off = mean_ut_off(lm, p.tab_bytes);
    const uint32_t ut_bytes = mean_ut_bytes(T);
    const uint32_t lz_off = ut_off + 2u * ut_bytes;
    float *bins = reinterpret_cast<float *>(smem_raw + bins_off);

    for (int t = tid; t < lm; t += kThreads) bins[t] = 0.f;
    if (tid < 2 * kListPadRows)
        reinterpret_cast<float *>(smem_raw + ut_off + (size_t)(tid / kListPadRows) * ut_bytes)[T + tid % kListPadRows] = 0.f;
    if (tid < 2) ctr[tid] = 0;
    if (tid < kPW * 2) sums[tid] = 0.0;
    __syncthreads();
    fda_grid_wait();

    const int64_t n_tiles = p.tiles > c ? (p.tiles - c + p.cpg - 1) / p.cpg : 0;

    if (warp < kPW) {
        // =============================== producers ===============================
        const int pt = tid;                                   // quad of indices inside a batch
        float nf = 0.f, pf = 0.f;
        // head of the schedule record of the tile being stored (the walkers' item table) and the
        // record offsets of the next tile, loaded one and two tiles ahead of their use
        uint4 tabv = make_uint4(0u, 0u, 0u, 0u);
        unsigned long long off0 = load_u64(p.sched_off + c), off1 = load_u64(p.sched_off + c + 1);
        if (pt * 16 < p.tab_bytes) tabv = load_u4(p.sched + off0 + pt * 16);
        if (pt == 0) rec_off[0] = off0;
        if (n_tiles > 1) { off0 = load_u64(p.sched_off + c + p.cpg); off1 = load_u64(p.sched_off + c + p.cpg + 1); }

        // Slot s, row r: lz + (s * R + r) * kRowPitch, a thread's 16 bytes of it.  A slot
        // holds up to rp rows of w; the slot of a quad's first rows also w_t0 and xi, behind them.
        const int D = mp.depth, rp = MULTI ? mp.piece : p.K;
        const int R = rp + 1 + (LINEAR ? 1 : 0);
        const uint32_t lz = smem_base + lz_off + (uint32_t)pt * 16u;
        int left_i = (int)n_tiles * p.nb;                     // quads of this thread that are still to be asked for,
        int b_i = 0, k_i = 0;                                 // the next one's batch in the tile and first row
        uint32_t j_i = (uint32_t)c * (uint32_t)T + 4u * pt;
        const uint32_t wrap = (uint32_t)(p.cpg - 1) * (uint32_t)T;   // from the end of a tile to this block's next one
        // n rows from `row` on into a slot
        auto copy = [&](uint32_t dst, const float *row, int n) {
            const float *q = row + j_i;
            if (VEC) {
                if (j_i + 4u <= (uint32_t)p.d) {
#pragma unroll 4
                    for (int k = 0; k < n; ++k) cp_async16(dst + (uint32_t)k * kRowPitch, q + (int64_t)k * p.row_stride);
                } else {                                       // the end of the model
#pragma unroll 1
                    for (int k = 0; k < n; ++k, q += p.row_stride, dst += kRowPitch)
#pragma unroll
                        for (uint32_t e = 0; e < 4; ++e) cp_async4(dst + 4u * e, j_i + e < (uint32_t)p.d ? q + e : row, j_i + e < (uint32_t)p.d);
                }
            } else {
                // the warp's 128 indices, 32 consecutive ones at a time (a lane's quad is copied by other lanes)
                q -= 3 * lane;
                dst -= 12u * lane;
                const uint32_t j0 = j_i - 3u * lane;
#pragma unroll 1
                for (int k = 0; k < n; ++k, q += p.row_stride, dst += kRowPitch)
#pragma unroll
                    for (uint32_t e = 0; e < 128; e += 32) {
                        const bool on = j0 + e < (uint32_t)p.d;
                        cp_async4(dst + 4u * e, on ? q + e : row, on);
                    }
            }
        };
        auto issue = [&](int slot) {
            if (left_i > 0) {
                uint32_t dst = lz + (uint32_t)(slot * R) * kRowPitch;
                copy(dst, p.w + (int64_t)k_i * p.row_stride, MULTI ? min(rp, p.K - k_i) : rp);
                if (k_i == 0) {
                    dst += (uint32_t)rp * kRowPitch;
                    copy(dst, p.w_t0, 1);
                    if (LINEAR) copy(dst + kRowPitch, p.xi, 1);
                }
                if (MULTI) k_i += rp;
                if (!MULTI || k_i >= p.K) {
                    k_i = 0;
                    --left_i;
                    j_i += kBatch;
                    if (++b_i == p.nb) { b_i = 0; j_i += wrap; }
                }
            }
            cp_async_commit();                                 // (an empty group past the end keeps the count)
        };
        for (int s = 0; s < D; ++s) issue(s);
        int slot = 0;
        for (int64_t n = 0; n < n_tiles; ++n) {
            const int buf = (int)(n & 1);
            for (int b = 0; b < p.nb; ++b) {
                float4 w0 = make_float4(0.f, 0.f, 0.f, 0.f), x = w0, a = w0;
                float qn = 0.f;
                for (int k0 = 0; k0 < p.K; k0 += rp) {
                    cp_async_wait_upto(D - 1);                 // the oldest group has landed
                    if (!VEC) __syncwarp();                    // (all lanes' parts of it)
                    const uint32_t src = lz + (uint32_t)(slot * R) * kRowPitch;
                    if (k0 == 0) {
                        const uint32_t q = src + (uint32_t)rp * kRowPitch;
                        w0 = lds128(q);
                        if (LINEAR) x = lds128(q + kRowPitch);
                    }
                    const int m = MULTI ? min(rp, p.K - k0) : rp;
#pragma unroll 4
                    for (int k = 0; k < m; ++k) {
                        const float4 v = lds128(src + (uint32_t)k * kRowPitch);
                        const float ux = v.x - w0.x, uy = v.y - w0.y, uz = v.z - w0.z, uw = v.w - w0.w;
                        qn = fmaf(ux, ux, qn); qn = fmaf(uy, uy, qn);
                        qn = fmaf(uz, uz, qn); qn = fmaf(uw, uw, qn);
                        a.x += ux; a.y += uy; a.z += uz; a.w += uw;
                    }
                    if (!VEC) __syncwarp();                    // (read by all lanes)
                    issue(slot);                               // the slot is free again
                    slot = slot + 1 == D ? 0 : slot + 1;
                    if (!MULTI) break;
                }
                nf += qn;
                if (LINEAR) {
                    pf = fmaf(x.x, a.x, pf); pf = fmaf(x.y, a.y, pf);
                    pf = fmaf(x.z, a.z, pf); pf = fmaf(x.w, a.w, pf);
                }
                // rows 4*pt .. 4*pt+3 of the batch; row r is stored at r ^ ((r >> 3) & 3) (the
                // schedule's entries hold that row): one 16-byte store of the quad, its floats permuted
                const uint32_t r0 = (uint32_t)(b * kBatch + 4 * pt);
                const int sw = (int)((r0 >> 3) & 3u);
                store_row(smem_base + ut_off + (uint32_t)buf * ut_bytes + r0 * 4u,
                          comp(a, 0 ^ sw), comp(a, 1 ^ sw), comp(a, 2 ^ sw), comp(a, 3 ^ sw));
            }
            // ---- the tile is stored: its sums, its item table, its counter, then the hand-over ----
            // (fp32 within the tile: a thread's few indices, then the warp's tree; fp64 across tiles)
            {
                float sa = nf, sb = LINEAR ? pf : 0.f;
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) {
                    sa += __shfl_xor_sync(0xffffffffu, sa, off);
                    if (LINEAR) sb += __shfl_xor_sync(0xffffffffu, sb, off);
                }
                if (lane == 0) {
                    sums[warp * 2 + 0] += (double)sa;
                    if (LINEAR) sums[warp * 2 + 1] += (double)sb;
                }
                nf = 0.f; pf = 0.f;
            }
            // the table of this tile (loaded a tile ago), the loads of the next one, the offsets of
            // the one after: nothing here waits for memory
            if (pt * 16 < p.tab_bytes)
                *reinterpret_cast<uint4 *>(smem_raw + tab_off + (size_t)buf * p.tab_bytes + pt * 16) = tabv;
            if (pt == 0) { ctr[buf] = kWW; rec_off[(n + 1) & 3] = off0; }
            if (n + 1 < n_tiles) {
                const unsigned char *nrec = p.sched + off0;
                if (pt * 16 < p.tab_bytes) tabv = load_u4(nrec + pt * 16);
                for (uint64_t o = (uint64_t)pt * 128u; o < off1 - off0; o += (uint64_t)kPW * 32u * 128u)   // the record into L2 ahead of its walk
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(nrec + o));
            }
            if (n + 2 < n_tiles) {
                const int64_t t2 = c + (n + 2) * p.cpg;
                off0 = load_u64(p.sched_off + t2);
                off1 = load_u64(p.sched_off + t2 + 1);
            }
            block_barrier<kThreads>();
        }
        cp_async_wait_upto(0);
    } else {
        // =============================== walkers ===============================
        for (int64_t n = 0; n < n_tiles; ++n) {
            block_barrier<kThreads>();                                   // tile n is stored, tile n - 1 is walked
            const int buf = (int)(n & 1);
            const unsigned char *rec = p.sched + rec_off[n & 3];
            const uint32_t *tab = reinterpret_cast<const uint32_t *>(smem_raw + tab_off + (size_t)buf * p.tab_bytes);
            const int n_items = (int)tab[0];
            const uint16_t *cells = reinterpret_cast<const uint16_t *>(rec + fda_sched_cells_off(n_items));
            const unsigned char *ent0 = rec + fda_sched_entries_off(n_items);
            const uint32_t base = smem_base + ut_off + (uint32_t)buf * ut_bytes;
            // the first kWW items go to the warps in order, the others to whoever asks next
            int it = warp - kPW;
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
                float a = 0.f;
                // all entry loads of (up to) AHEAD chunks first, then the walk
                for (int c0 = 0; c0 < nch; c0 += AHEAD) {
                    uint2 ch[AHEAD];
#pragma unroll
                    for (int q = 0; q < AHEAD; ++q)
                        if (c0 + q < nch) ch[q] = __ldg(ent + (size_t)(c0 + q) * kListSlots);
#pragma unroll
                    for (int q = 0; q < AHEAD; ++q) gather1_chunk(ch[q], steps - 4 * (c0 + q), base, a);
                }
                flush1(bins, lm, cell, a);
            }
        }
    }
    block_barrier<kThreads>();                                           // the last tile is walked

    // ---- flush: bins -> this block's partial sketch; the producer warps' sums, in warp order ----
    {
        float *out = p.part_sk + (size_t)blockIdx.x * (size_t)lm;
        for (int t = tid; t < lm; t += kThreads) out[t] = bins[t];
    }
    if (tid < 2) {
        double t = 0.0;
        for (int q = 0; q < kPW; ++q) t += sums[q * 2 + tid];
        p.part_np[(size_t)blockIdx.x * 2 + tid] = t;
    }
}

// The sketch of one vector, the averaged drifts: no roles and no second buffer, a block's warps form its tile (24 KB, loaded
// a tile ahead), then walk.  p.part_tiles blocks share a tile, each walking every p.part_tiles-th item; a block serves one part
// of the sketch rows.
// Bound: latency.  A row of the tile is one float, so a tile is formed in one round trip and walked in a few thousand
// cycles; two small blocks to an SM cover each other's round trips, and a short vector gets more blocks than it has tiles.
// The first item's entries are asked for in front of fda_grid_wait (the schedule is older than the kernel before this one).
// Measured, all kernels of the averaged state back to back, K = 20, odd d, against 8 producer and 24 walker warps that served
// this vector, too: 7 x 500 16.7 -> 12.4 us (d = 60K), 20.3 -> 19.1 (500K), 43.3 -> 38.8 (1.2M), 443 -> 437 (20M); 8 x 1000 in
// parts, which are one launch now, 26.2 -> 12.4, 29.8 -> 21.1, 62.5 -> 49.9, 256 -> 243 (8M).  16 warps and two blocks to an
// SM are the best of 8 / 4, 12 / 2, 16 / 1, 16 / 2 and 24 / 1 or within 5 % of it.
constexpr int kShortWarps = 16, kShortPerSm = 2;
constexpr int kShortQuads = (kListMaxTile / 4 + kShortWarps * 32 - 1) / (kShortWarps * 32);
inline size_t mean_short_smem(int lm, int T) { return (size_t)align128((uint32_t)lm * 4u) + (size_t)(T + kListPadRows) * 4; }

__global__ void __launch_bounds__(kShortWarps * 32, kShortPerSm) k_mean_sketch_short(const ListParams p)
{
    constexpr int kThreads = kShortWarps * 32, kAhead = 7;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int split = p.part_tiles, T = p.T, lm = p.l * p.m, tiles = (int)p.tiles;
    // block = (sub * parts + part) * cpg + c: the tiles c, c + cpg, ...
    const int c = (int)blockIdx.x % p.cpg, part = (int)blockIdx.x / p.cpg % p.groups, sub = (int)blockIdx.x / (p.cpg * p.groups);
    const uint32_t ut_off = align128((uint32_t)lm * 4u), base = (uint32_t)__cvta_generic_to_shared(smem_raw) + ut_off;
    float *bins = reinterpret_cast<float *>(smem_raw);

    const uint64_t *sched_off = p.sched_off + (size_t)part * p.nb;
    const uint32_t *tab = nullptr;
    const uint16_t *cells = nullptr;
    const unsigned char *ent0 = nullptr;
    int it = 0, n_items = 0, steps = 0;
    uint32_t cell = 0;
    const uint2 *ent = nullptr;
    uint2 ch[kAhead];
    auto ask = [&](int first) {                               // the chunks first .. first + kAhead - 1 of the item
#pragma unroll
        for (int q = 0; q < kAhead; ++q)
            if (4 * (first + q) < steps) ch[q] = __ldg(ent + (size_t)(first + q) * kListSlots);
    };
    auto fetch = [&]() {
        const uint32_t d0 = __ldg(tab + 4 + 2 * it), chunk0 = __ldg(tab + 5 + 2 * it);
        steps = (int)(d0 & 0xffffu);
        cell = __ldg(cells + (size_t)(d0 >> 16) * kListSlots + lane);
        ent = reinterpret_cast<const uint2 *>(ent0 + (size_t)chunk0 * 256) + lane;
        ask(0);
    };
    auto open_tile = [&](int t) {
        const unsigned char *rec = p.sched + load_u64(sched_off + t);
        tab = reinterpret_cast<const uint32_t *>(rec);
        n_items = (int)__ldg(tab);
        cells = reinterpret_cast<const uint16_t *>(rec + fda_sched_cells_off(n_items));
        ent0 = rec + fda_sched_entries_off(n_items);
        it = warp * split + sub;
        if (it < n_items) fetch();
    };
    float4 v[kShortQuads];
    auto load_tile = [&](int t) {
#pragma unroll
        for (int u = 0; u < kShortQuads; ++u) {
            const int q = tid + u * kThreads;
            const int64_t j = (int64_t)t * T + 4 * q, left = q < T / 4 ? p.d - j : 0;
            v[u] = load_quad<false>(p.w + j, left >= 4, left > 0 ? (int)left : 0);
        }
    };
    open_tile(c);
    for (int t = tid; t < lm; t += kThreads) bins[t] = 0.f;
    if (tid < kListPadRows) reinterpret_cast<float *>(smem_raw + ut_off)[T + tid] = 0.f;
    fda_grid_wait();
    load_tile(c);
    for (int t = c; t < tiles; t += p.cpg) {
#pragma unroll
        for (int u = 0; u < kShortQuads; ++u) {               // row r of the tile at r ^ ((r >> 3) & 3): the quad's floats permuted
            const int q = tid + u * kThreads, sw = (q >> 1) & 3;
            if (q < T / 4) store_row(base + 16u * q, comp(v[u], 0 ^ sw), comp(v[u], 1 ^ sw), comp(v[u], 2 ^ sw), comp(v[u], 3 ^ sw));
        }
        __syncthreads();
        const bool more = t + p.cpg < tiles;
        if (more) load_tile(t + p.cpg);
        while (it < n_items) {
            float a = 0.f;
            for (int c0 = 0;;) {
#pragma unroll
                for (int q = 0; q < kAhead; ++q) gather1_chunk(ch[q], steps - 4 * (c0 + q), base, a);
                c0 += kAhead;
                if (4 * c0 >= steps) break;
                ask(c0);
            }
            const uint32_t done = cell;
            it += kShortWarps * split;
            if (it < n_items) fetch();
            flush1(bins, lm, done, a);
        }
        if (more) open_tile(t + p.cpg);
        __syncthreads();
    }
    float *out = p.part_sk + ((size_t)part * p.cpg * split + sub * p.cpg + c) * lm;
    for (int t = tid; t < lm; t += kThreads) out[t] = bins[t];
}

// Averaged state: mean_state[e] = (sum over the blocks of the partials) / divisor, in fp64 and in a
// fixed order.  Block 0 takes the two scalars, from part_np[b * 2 + e], b < np_blocks - the partials of
// the list kernel or of the pass that averaged the drifts - and divides them by K; every other block 32
// cells, eight threads to a cell.  Bound: latency, so twelve loads are in flight per thread.  Averaged
// state with K = 10, d = 1.2M (148 blocks, 1172 pairs), back to back: 36.4 -> 28.9 us, d = 61,706, K = 5
// 15.3 -> 12.5 us, against one thread per cell and one warp per scalar.
constexpr int kFinalThreads = 256, kFinalCells = 32, kFinalLoads = 12;

template <typename T>
__device__ __forceinline__ double sum_strided(const T *src, int first, int step, int n, size_t pitch)
{
    double acc = 0.0;
    for (int b = first; b < n; b += kFinalLoads * step) {
        T v[kFinalLoads];
#pragma unroll
        for (int u = 0; u < kFinalLoads; ++u) v[u] = src[(size_t)(b + u * step < n ? b + u * step : b) * pitch];
#pragma unroll
        for (int u = 0; u < kFinalLoads; ++u) acc += b + u * step < n ? (double)v[u] : 0.0;
    }
    return acc;
}

__global__ void __launch_bounds__(kFinalThreads)
k_finalize_mean(const float *part_sk, const double *part_np, int blocks, int np_blocks, int cells, int lm /* of a part */,
                int K, uint32_t flags, bool have_xi, double cell_div, float *mean_state)
{
    __shared__ double red[kFinalThreads];
    const int tid = threadIdx.x;
    fda_grid_wait();
    if (blockIdx.x == 0) {
        const int e = tid & 1;
        const bool on = e == 0 ? (flags & FDA_STATE_NORM) != 0 : ((flags & FDA_STATE_LINEAR) != 0 && have_xi);
        red[tid] = on ? sum_strided(part_np + e, tid >> 1, kFinalThreads / 2, np_blocks, 2) : 0.0;
        __syncthreads();
        if (tid < 64) {                         // warp e adds the values of scalar e
            double acc = 0.0;
            for (int q = tid & 31; q < kFinalThreads / 2; q += 32) acc += red[2 * q + (tid >> 5)];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            if ((tid & 31) == 0) mean_state[tid >> 5] = (float)(acc / (double)K);
        }
        return;
    }
    const int cell = ((int)blockIdx.x - 1) * kFinalCells + tid % kFinalCells, slice = tid / kFinalCells;
    constexpr int kSlices = kFinalThreads / kFinalCells;
    double acc = 0.0;
    if (cell < cells && (flags & FDA_STATE_SKETCH))
        acc = sum_strided(part_sk + (size_t)(cell / lm) * blocks * lm + cell % lm, slice, kSlices, blocks, (size_t)lm);
    red[tid] = acc;
    __syncthreads();
    if (slice == 0 && cell < cells) {
        double t = 0.0;
#pragma unroll
        for (int q = 0; q < kSlices; ++q) t += red[q * kFinalCells + tid];
        mean_state[2 + cell] = (float)(t / cell_div);
    }
}

template <int AHEAD>
void (*pick_kernel(bool linear, bool multi, bool vec))(MeanParams)
{
    if (!vec) return linear ? k_mean_state_gather<true, AHEAD, true, false> : k_mean_state_gather<false, AHEAD, true, false>;
    if (multi) return linear ? k_mean_state_gather<true, AHEAD, true, true> : k_mean_state_gather<false, AHEAD, true, true>;
    return linear ? k_mean_state_gather<true, AHEAD, false, true> : k_mean_state_gather<false, AHEAD, false, true>;
}

// What both passes need of the context and the call (l, m: of a part of the sketch rows)
ListParams mean_params(const fda_ctx *ctx, const float *w, int64_t row_stride, int K, int64_t d)
{
    ListParams p{};
    p.w = w; p.row_stride = row_stride; p.K = K; p.d = d;
    p.l = ctx->l / ctx->sched_parts; p.m = ctx->m;
    p.T = ctx->sched_T;
    p.sched = ctx->sched; p.sched_off = ctx->sched_off;
    p.part_sk = ctx->part_sk; p.part_np = ctx->part_np;
    p.tiles = (d + p.T - 1) / p.T;
    return p;
}

}  // namespace

// mean_state from the partial sums: `blocks` partial sketches per part of lm cells, np_blocks partial pairs.
cudaError_t fda_launch_finalize_mean(const fda_ctx *ctx, int blocks, int np_blocks, int lm, int K, uint32_t flags,
                                     bool have_xi, double cell_div, float *mean_state, cudaStream_t s)
{
    return fda_launch_dependent(k_finalize_mean, 1 + (ctx->lm + kFinalCells - 1) / kFinalCells, kFinalThreads, 0, s,
                                ctx->part_sk, ctx->part_np, blocks, np_blocks, ctx->lm, lm, K, flags, have_xi, cell_div,
                                mean_state);
}

// The averaged state S-bar of fda_mean_state in one pass over the K rows.  Returns
// cudaErrorNotSupported when the request does not fit this path (the caller then uses the other
// kernels); any other value is the result of the launches.
cudaError_t fda_launch_mean_state_gather(fda_ctx *ctx, const float *w, int64_t row_stride, int K,
                                         int64_t d, const float *w_t0, const float *xi,
                                         uint32_t flags, float *mean_state, cudaStream_t s)
{
    if (!(flags & FDA_STATE_SKETCH) || ctx->l == 0 || !ctx->sched) return cudaErrorNotSupported;
    const float *xi_used = (flags & FDA_STATE_LINEAR) ? xi : nullptr;
    if (ctx->sched_parts > 1) return cudaErrorNotSupported;         // every part would read the K rows again

    MeanParams mp{};
    ListParams &p = mp.q;
    p = mean_params(ctx, w, row_stride, K, d);
    p.w_t0 = w_t0; p.xi = xi_used; p.have_xi = xi_used != nullptr;
    p.vec = ((((uintptr_t)w | (uintptr_t)w_t0 | (uintptr_t)(xi_used ? xi_used : w)) & 15u) == 0) && (row_stride % 4 == 0);
    p.tab_bytes = fda_list_table_bytes(ctx->sched_ni_max);
    p.groups = 1;
    p.cpg = (int)std::min((int64_t)ctx->n_sm, p.tiles);
    const int blocks = p.cpg, lm = ctx->lm;
    if ((size_t)blocks * lm > ctx->part_sk_floats || blocks > ctx->max_blocks || (size_t)blocks * 2 > ctx->part_np_doubles)
        return cudaErrorNotSupported;
    if (p.T % kBatch != 0 || kPW * 32 * 16 < p.tab_bytes) return cudaErrorNotSupported;
    p.nb = p.T / kBatch;
    // what the single-column tile leaves free becomes the producers' landing zone
    const size_t fixed = mean_smem_fixed(p.l, p.m, p.T, p.tab_bytes);
    // (up to kMaxPiece rows arrive in one slot, more of them in several of nearly equal size)
    const int slots = (K + kMaxPiece - 1) / kMaxPiece;
    mp.piece = (K + slots - 1) / slots;
    const size_t per_slot = (size_t)kRowPitch * (size_t)(mp.piece + 1 + (xi_used ? 1 : 0));
    const size_t depth = (size_t)ctx->smem_optin > fixed ? ((size_t)ctx->smem_optin - fixed) / per_slot : 0;
    // too little room to keep three slots per thread in flight: the pass would wait for its loads
    if (depth < 3) return cudaErrorNotSupported;
    mp.depth = (int)(depth < (size_t)kMaxDepth ? depth : (size_t)kMaxDepth);
    const size_t smem = fixed + (size_t)mp.depth * per_slot;

    auto kern = p.l >= 7 ? pick_kernel<5>(xi_used != nullptr, slots > 1, p.vec != 0)
                         : pick_kernel<kChunksAhead>(xi_used != nullptr, slots > 1, p.vec != 0);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ctx->smem_optin);
    if (e == cudaSuccess) e = fda_launch_dependent(kern, blocks, kThreads, smem, s, mp);
    if (e != cudaSuccess) return e;
    return fda_launch_finalize_mean(ctx, blocks, blocks, lm, K, flags, xi_used != nullptr, (double)K, mean_state, s);
}

// The cells of S-bar from the vector of averaged drifts (d floats, 16-byte aligned), the scalars
// from the np_blocks partial pairs at the start of ctx->part_np; same return convention.
cudaError_t fda_launch_mean_sketch_gather(fda_ctx *ctx, const float *mean_drift, int K, int64_t d, bool have_xi,
                                          uint32_t flags, int np_blocks, float *mean_state, cudaStream_t s)
{
    if (!(flags & FDA_STATE_SKETCH) || ctx->l == 0 || !ctx->sched) return cudaErrorNotSupported;
    ListParams p = mean_params(ctx, mean_drift, 0, 1, d);
    const int parts = ctx->sched_parts, lm = p.l * p.m;
    p.groups = parts;
    p.nb = (int)ctx->sched_tiles;                                    // records of a part
    p.cpg = (int)std::max((int64_t)1, std::min((int64_t)ctx->n_sm * kShortPerSm / parts, p.tiles));
    // up to three blocks to a tile while each has an SM of its own, two to an SM where a warp has six items or more to walk.  Measured, whole
    // calls, one block to a tile and two, K = 24: 7 x 500 (seven items) d = 400K 21.4 and 21.1 us, 480K 23.8 and 22.7, 612K 31.3 and 29.5, 700K
    // 34.4 and 32.1; 8 x 1000, K = 20, d = 200K (eight) 18.3 and 16.8, 360K 20.1 and 19.4; but 5 x 250 (three) d = 480K 19.6 and 20.3, K = 8,
    // d = 800K 17.2 and 18.4; 10 x 250, K = 12, d = 600K (five) 19.3 and 20.1.
    const bool long_walk = p.l * ((p.m + kListSlots - 1) / kListSlots) >= 6 * kShortWarps && p.tiles * parts > ctx->n_sm / 2;
    p.part_tiles = (int)std::max((int64_t)1, std::min((int64_t)3, (long_walk ? kShortPerSm : 1) * ctx->n_sm / (p.tiles * parts)));
    const int n = p.cpg * p.part_tiles;                              // partial sketches of a part
    const size_t smem = mean_short_smem(lm, p.T);
    if ((size_t)n * lm * parts > ctx->part_sk_floats || p.T > kShortQuads * kShortWarps * 32 * 4 || smem > (size_t)ctx->smem_optin)
        return cudaErrorNotSupported;
    cudaError_t e = cudaFuncSetAttribute(k_mean_sketch_short, cudaFuncAttributeMaxDynamicSharedMemorySize, ctx->smem_optin);
    if (e == cudaSuccess) e = fda_launch_dependent(k_mean_sketch_short, n * parts, kShortWarps * 32, smem, s, p);
    if (e != cudaSuccess) return e;
    return fda_launch_finalize_mean(ctx, n, np_blocks, lm, K, flags, have_xi, 1.0, mean_state, s);
}
