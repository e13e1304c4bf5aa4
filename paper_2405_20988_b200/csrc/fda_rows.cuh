// Streaming pass over the rows of w for ||u^(k)||^2 and <xi,u^(k)> (Section 3, local state;
// Section 3.2, LinearFDA), shared by fda_local_state_linear.cu and fda_noalloc.cu.
//
// Bound: HBM (K*d + 2*d floats are read once, K pairs written).  A block serves a group of at most
// five rows and a strided set of 1024-index chunks; a thread takes one quad of indices of a chunk,
// asks for the quad of all its rows, of w_t0 and of xi before it uses any, and keeps the 2 x 5 sums
// in fp64 registers (a quad is summed in fp32 first), so nothing is staged in shared memory and no
// barrier stands in the loop.  w_t0 and xi are read once per group; the blocks of the groups are
// interleaved over the same chunks, so those reads hit L2.
//
// Rows need not be 16-byte aligned.  Only the sums over a row are wanted, so every row is cut into
// quads at its own 16-byte boundaries: the quad q of row k covers indices c0 + r_k + 4q .. + 3, where
// c0 is the first index at which w_t0 is aligned and r_k in 0..3 the distance to the row's own
// boundary.  All row loads stay 128-bit; w_t0 and xi are read as two neighbouring quads (the second
// hits L1) from which the row picks its four values.  What the quads do not cover - up to six
// indices in front and up to eleven at the end - one block per group adds with 32-bit loads.
// Measured on B200 (K = 30, d = 6,964,106, with xi, the pass alone): 150 us with aligned rows and
// 160 us at a pitch of d, 6.0 and 5.6 TB/s.  Eight rows a block at two blocks per SM (the sums leave
// 128 registers): 150 and 171 us; four rows, four blocks: 150 and 182 us.  The kernel before it (32-bit loads for rows that are not aligned): 226 us.
#ifndef FDA_ROWS_CUH_
#define FDA_ROWS_CUH_

#include "fda_internal.h"
#include "fda_quads.cuh"

namespace fda_rows {

using fda_quads::first_aligned;
using fda_quads::pick;

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kRows = 5;              // rows of a group: 2 * kRows fp64 sums in registers
constexpr int kBlocksPerSm = 3;
constexpr int kVals = 16;             // partial sums of a block: (norm, projection) per row, then zeros
static_assert(kWarps >= kRows && kVals >= 2 * kRows, "the uncovered ends of row k are added by warp k");

struct Params {
    const float *w, *w_t0, *xi;       // xi null: no projection
    int64_t row_stride, d;
    int K;
    int groups, cpg;                  // block = c * groups + g
    int slen;                         // floats of a state (2 + sketch cells, which are written as 0)
    uint32_t flags;
    double *part;                     // [block][kVals]
    unsigned int *ticket;             // [groups], 0 between launches (fused finish only)
    float *states;
};

// rows [first, first + n) of group g: K / groups each, one more in the first K % groups
__device__ __forceinline__ int group_first(const Params &p, int g)
{
    const int base = p.K / p.groups, more = p.K % p.groups;
    return g * base + (g < more ? g : more);
}
__device__ __forceinline__ int group_rows(const Params &p, int g) { return p.K / p.groups + (g < p.K % p.groups ? 1 : 0); }

// Adds the pairs of all blocks of group g in a fixed order (16 threads per value, then their sums in
// order) and writes the rows' states.  Called by one block; red: kThreads doubles of shared memory.
__device__ __forceinline__ void finish_group(const Params &p, int g, double *red)
{
    const int tid = threadIdx.x, e = tid % kVals, sl = tid / kVals;
    constexpr int kSlices = kThreads / kVals;
    double t = 0.0;
    for (int b = sl; b < p.cpg; b += kSlices) t += __ldcg(p.part + ((size_t)b * p.groups + g) * kVals + e);
    red[tid] = t;
    __syncthreads();
    if (tid < kVals) {
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < kSlices; ++q) s += red[q * kVals + tid];
        const int k = tid >> 1;
        const bool on = (tid & 1) == 0 ? (p.flags & FDA_STATE_NORM) != 0 : p.xi != nullptr;
        if (k < group_rows(p, g)) p.states[(size_t)(group_first(p, g) + k) * p.slen + (tid & 1)] = on ? (float)s : 0.f;
    }
}

// Ordinary loads, not ld.global.nc: the kernel before this one may have written what they read (fda_launch_dependent).
__device__ __forceinline__ float4 load4(const float *ptr) { return *reinterpret_cast<const float4 *>(ptr); }
__device__ __forceinline__ float4 load4_any(const float *ptr)
{
    return make_float4(ptr[0], ptr[1], ptr[2], ptr[3]);
}

// XI: 0 no projection, 1 xi is aligned like w_t0, 2 it is not.  SHIFT: some row is not aligned like w_t0.  FUSED: the last block of a group writes the
// group's states (a ticket per group, no waiting); otherwise a second kernel calls finish_group.
template <int XI, bool SHIFT, bool FUSED>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm) k_rows_state(const Params p)
{
    constexpr bool LINEAR = XI != 0;
    __shared__ double red[kThreads];
    __shared__ bool last_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = (int)blockIdx.x % p.groups, c = (int)blockIdx.x / p.groups;
    const int first = group_first(p, g), n = group_rows(p, g);
    const float *wg = p.w + (size_t)first * (size_t)p.row_stride;

    const int c0 = first_aligned(p.w_t0);                     // first index at which w_t0 is aligned
    unsigned rs = 0;                                          // r_k of the rows, two bits each
#pragma unroll
    for (int k = 0; k < kRows; ++k)
        rs |= (unsigned)first_aligned(wg + c0 + (int64_t)(k < n ? k : 0) * p.row_stride) << (2 * k);
    fda_grid_wait();
    // quads whose two-quad window lies inside the vectors
    const int64_t Q = p.d >= c0 + 8 ? (p.d - 8 - c0) / 4 + 1 : 0;

    double acc[kVals];
#pragma unroll
    for (int e = 0; e < kVals; ++e) acc[e] = 0.0;

    const float *w0 = p.w_t0 + c0, *xi = LINEAR ? p.xi + c0 : nullptr;
    for (int64_t q = (int64_t)c * kThreads + tid; q < Q; q += (int64_t)p.cpg * kThreads) {
        const float *wq = wg + c0 + 4 * q;
        float4 a[kRows], x0, x1, b0, b1;
        b0 = load4(w0 + 4 * q);
        if (SHIFT) b1 = load4(w0 + 4 * q + 4);
        if (LINEAR) {
            x0 = XI == 1 ? load4(xi + 4 * q) : load4_any(xi + 4 * q);
            if (SHIFT) x1 = XI == 1 ? load4(xi + 4 * q + 4) : load4_any(xi + 4 * q + 4);
        }
        // (a group short of five rows repeats its first one: predicated loads ran 9 % slower)
#pragma unroll
        for (int k = 0; k < kRows; ++k)
            a[k] = __ldcs(reinterpret_cast<const float4 *>(wq + (int64_t)(k < n ? k : 0) * p.row_stride + (SHIFT ? (rs >> (2 * k)) & 3u : 0u)));
#pragma unroll
        for (int k = 0; k < kRows; ++k) {
            if (k >= n) continue;
            const int r = SHIFT ? (int)((rs >> (2 * k)) & 3u) : 0;
            const float4 b = SHIFT ? pick(b0, b1, r) : b0;
            const float ux = a[k].x - b.x, uy = a[k].y - b.y, uz = a[k].z - b.z, uw = a[k].w - b.w;
            acc[2 * k] += (double)fmaf(uw, uw, fmaf(uz, uz, fmaf(uy, uy, ux * ux)));
            if (LINEAR) {
                const float4 x = SHIFT ? pick(x0, x1, r) : x0;
                acc[2 * k + 1] += (double)fmaf(x.w, uw, fmaf(x.z, uz, fmaf(x.y, uy, x.x * ux)));
            }
        }
    }

    // the 16 values of a warp: in each of four steps a lane gives away half of the sums it holds and
    // adds its partner's halves of the others; lanes 2e and 2e + 1 end with value e
#pragma unroll
    for (int off = 16, cnt = kVals / 2; cnt >= 1; off >>= 1, cnt >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < kVals / 2; ++i)
            if (i < cnt) {
                const double send = up ? acc[i] : acc[i + cnt], keep = up ? acc[i + cnt] : acc[i];
                acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
            }
    }
    double v = acc[0] + __shfl_xor_sync(0xffffffffu, acc[0], 1);
    if ((lane & 1) == 0) red[warp * kVals + (lane >> 1)] = v;

    // block c = 0 of the group: the ends of row k, one warp per row
    double en = 0.0, ep = 0.0;
    if (c == 0 && warp < n) {
        const int head = (int)min(p.d, (int64_t)(c0 + ((rs >> (2 * warp)) & 3u)));
        const int64_t tail = Q > 0 ? c0 + (int64_t)((rs >> (2 * warp)) & 3u) + 4 * Q : head;
        const int64_t j = lane < head ? lane : tail + (lane - head);
        if (j < p.d) {
            const float u = wg[(int64_t)warp * p.row_stride + j] - p.w_t0[j];
            en = (double)(u * u);
            if (LINEAR) ep = (double)(p.xi[j] * u);
        }
    }
    if (c == 0) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            en += __shfl_xor_sync(0xffffffffu, en, off);
            ep += __shfl_xor_sync(0xffffffffu, ep, off);
        }
        if (lane == 0) { red[kWarps * kVals + 2 * warp] = en; red[kWarps * kVals + 2 * warp + 1] = ep; }   // zeros from the warps without a row
    }
    __syncthreads();
    if (tid < kVals) {
        double t = c == 0 ? red[kWarps * kVals + tid] : 0.0;
        for (int q = 0; q < kWarps; ++q) t += red[q * kVals + tid];
        p.part[(size_t)blockIdx.x * kVals + tid] = t;
    }
    // the cells of a context with a sketch that were not asked for
    if (p.slen > 2) {
        const int cells = p.slen - 2;
        for (int64_t t = (int64_t)c * kThreads + tid; t < (int64_t)n * cells; t += (int64_t)p.cpg * kThreads)
            p.states[(size_t)(first + t / cells) * p.slen + 2 + t % cells] = 0.f;
    }
    if (FUSED) {
        if (tid < kVals) __threadfence();
        __syncthreads();
        if (tid == 0) last_s = atomicAdd(p.ticket + g, 1u) == (unsigned)p.cpg - 1u;
        __syncthreads();
        if (!last_s) return;
        __threadfence();
        finish_group(p, g, red);
        if (tid == 0) p.ticket[g] = 0u;                       // ready for the next launch
    }
}

// blocks per group for a vector of d elements on n_sm SMs
inline int blocks_per_group(int n_sm, int groups, int64_t d)
{
    int64_t chunks = (d / 4 + kThreads - 1) / kThreads, cpg = (int64_t)n_sm * kBlocksPerSm / groups;
    if (cpg > chunks) cpg = chunks;
    return cpg < 1 ? 1 : (int)cpg;
}
// the kernel for the alignments of a call
template <bool FUSED>
inline void (*kernel_for(const Params &p))(Params)
{
    const unsigned a = (unsigned)((uintptr_t)p.w & 15u), b = (unsigned)((uintptr_t)p.w_t0 & 15u);
    const bool shift = a != b || (p.K > 1 && (p.row_stride & 3) != 0);
    const int xi = !p.xi ? 0 : ((unsigned)((uintptr_t)p.xi & 15u) == b ? 1 : 2);
    if (xi == 0) return shift ? k_rows_state<0, true, FUSED> : k_rows_state<0, false, FUSED>;
    if (xi == 1) return shift ? k_rows_state<1, true, FUSED> : k_rows_state<1, false, FUSED>;
    return shift ? k_rows_state<2, true, FUSED> : k_rows_state<2, false, FUSED>;
}

}  // namespace fda_rows

#endif
