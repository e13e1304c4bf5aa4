// Pieces shared by the two kernels that walk the list schedule (fda_sched.cu): the per-worker
// sketch pass (fda_local_state_gather.cu) and the averaged state (fda_mean_state_gather.cu).
#ifndef FDA_LIST_KERNEL_CUH_
#define FDA_LIST_KERNEL_CUH_

#include "fda_internal.h"

namespace fda_list {

constexpr int GW = kListWorkers;
constexpr int kChunksAhead = 8;                // entry chunks (four steps each) the walkers of the averaged state load ahead (long items)

struct ListParams {
    const float *w, *w_t0, *xi;
    int64_t row_stride;
    int K;
    int64_t d;
    int have_xi;
    int vec;                         // 16-byte aligned inputs: the producers load 128 bits at a time
    int l, m;                        // sketch rows of a part, columns
    int groups, cpg;                 // block = c * groups + g
    int wgroups;                     // worker groups: g = part * wgroups + worker group
    int part_tiles;                  // several parts: records of a part of the sketch rows;
                                     // one part: blocks that share the items of a tile
    int T, nb;                       // indices and batches per tile
    int64_t tiles;                   // tiles that hold indices below d
    int tab_bytes;                   // bytes of one item-table buffer in shared memory
    const unsigned char *sched;
    const uint64_t *sched_off;
    const uint32_t *lane_prog;         // cells that stay with their lanes (else null): see fda_ctx
    const int2 *lane_rows;
    int lane_items;
    float *part_sk;                  // [block][cell][GW]
    double *part_np;                 // [block][GW][2]
};

template <int THREADS>
__device__ __forceinline__ void block_barrier()
{
    asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
}

// Loads and stores of the producers as volatile statements: the compiler keeps them in program
// order, so a batch's loads are issued kDepth batches before its values are used.  What the kernel before
// this one may have written (w, w_t0, xi) is not read through ld.global.nc: see fda_launch_dependent.
__device__ __forceinline__ float4 load4_stream(const float *ptr)
{
    float4 v;
    asm volatile("ld.global.cs.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(ptr));
    return v;
}
__device__ __forceinline__ float4 load4_keep(const float *ptr)
{
    float4 v;
    asm volatile("ld.global.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(ptr));
    return v;
}
__device__ __forceinline__ float load1(const float *ptr, bool on)
{
    float v;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\tmov.b32 %0, 0;\n\t@p ld.global.f32 %0, [%1];\n\t}"
                 : "=f"(v) : "l"(ptr), "r"((int)on));
    return v;
}
// four floats from ptr: one 128-bit load when `vec` (aligned, all four below the end), else the
// `n` valid ones with 32-bit loads and zeros behind them
template <bool STREAM>
__device__ __forceinline__ float4 load_quad(const float *ptr, bool vec, int n)
{
    if (vec) return STREAM ? load4_stream(ptr) : load4_keep(ptr);
    float4 v;
    v.x = load1(ptr, n > 0); v.y = load1(ptr + 1, n > 1); v.z = load1(ptr + 2, n > 2); v.w = load1(ptr + 3, n > 3);
    return v;
}
// the first n of the four floats ptr, ptr + 32, ptr + 64, ptr + 96, zeros for the others
__device__ __forceinline__ float4 load_strided(const float *ptr, int n)
{
    float4 v;
    v.x = load1(ptr, n > 0); v.y = load1(ptr + 32, n > 1); v.z = load1(ptr + 64, n > 2); v.w = load1(ptr + 96, n > 3);
    return v;
}
__device__ __forceinline__ uint4 load_u4(const void *ptr)
{
    uint4 v;
    asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(ptr));
    return v;
}
__device__ __forceinline__ uint2 load_u2(const void *ptr)
{
    uint2 v;
    asm volatile("ld.global.nc.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(ptr));
    return v;
}
__device__ __forceinline__ unsigned long long load_u64(const void *ptr)
{
    unsigned long long v;
    asm volatile("ld.global.nc.u64 %0, [%1];" : "=l"(v) : "l"(ptr));
    return v;
}
__device__ __forceinline__ void store_row(uint32_t addr, float x, float y, float z, float w)
{
    asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}
__device__ __forceinline__ float comp(const float4 &v, int q) { return q == 0 ? v.x : (q == 1 ? v.y : (q == 2 ? v.z : v.w)); }

// One schedule entry: gather the row (four workers) and add it with the entry's sign.  The
// sums stay packed as fp32 pairs, the sign is a multiplication by (+-1, +-1) (exact).
__device__ __forceinline__ void gather_row(uint32_t row_off, uint32_t sign_one, uint32_t base,
                                           unsigned long long &a01, unsigned long long &a23)
{
    unsigned long long u0, u1, ss;
    asm volatile("ld.shared.v2.b64 {%0,%1}, [%2];" : "=l"(u0), "=l"(u1) : "r"(base + row_off));
    asm("mov.b64 %0, {%1,%1};" : "=l"(ss) : "r"(sign_one));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a01) : "l"(u0), "l"(ss));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a23) : "l"(u1), "l"(ss));
}
// low / high half of a 32-bit word holding two entries (bits 0..12 row, bit 15 sign)
__device__ __forceinline__ void gather_lo(uint32_t w, uint32_t base, unsigned long long &a01, unsigned long long &a23)
{
    gather_row((w & 0x1fffu) << 4, ((w << 16) & 0x80000000u) ^ 0x3f800000u, base, a01, a23);
}
__device__ __forceinline__ void gather_hi(uint32_t w, uint32_t base, unsigned long long &a01, unsigned long long &a23)
{
    gather_row((w >> 12) & 0x1fff0u, (w & 0x80000000u) ^ 0x3f800000u, base, a01, a23);
}

// one chunk of an item: the steps that are left of it, at most four
__device__ __forceinline__ void walk_chunk(const uint2 &ch, int left, uint32_t base, unsigned long long &a01, unsigned long long &a23)
{
    if (left >= 4) {
        gather_lo(ch.x, base, a01, a23);
        gather_hi(ch.x, base, a01, a23);
        gather_lo(ch.y, base, a01, a23);
        gather_hi(ch.y, base, a01, a23);
    } else if (left > 0) {
        gather_lo(ch.x, base, a01, a23);
        if (left > 1) gather_hi(ch.x, base, a01, a23);
        if (left > 2) gather_lo(ch.y, base, a01, a23);
    }
}
// two chunks: one block of code while eight steps are left
__device__ __forceinline__ void walk_chunks2(const uint2 &c0, const uint2 &c1, int left, uint32_t base, unsigned long long &a01, unsigned long long &a23)
{
    if (left >= 8) {
        gather_lo(c0.x, base, a01, a23);
        gather_hi(c0.x, base, a01, a23);
        gather_lo(c0.y, base, a01, a23);
        gather_hi(c0.y, base, a01, a23);
        gather_lo(c1.x, base, a01, a23);
        gather_hi(c1.x, base, a01, a23);
        gather_lo(c1.y, base, a01, a23);
        gather_hi(c1.y, base, a01, a23);
    } else { walk_chunk(c0, left, base, a01, a23); walk_chunk(c1, left - 4, base, a01, a23); }
}
// the sums of an item's 32 lists into the bins
__device__ __forceinline__ void flush_item(float *bins, int lm, uint32_t cell, unsigned long long a01, unsigned long long a23)
{
    float4 acc;
    asm("mov.b64 {%0,%1}, %2;" : "=f"(acc.x), "=f"(acc.y) : "l"(a01));
    asm("mov.b64 {%0,%1}, %2;" : "=f"(acc.z), "=f"(acc.w) : "l"(a23));
    if ((cell & 0x7fffu) < (uint32_t)lm) {
        float *b = bins + (cell & 0x7fffu) * GW;
        if (cell & 0x8000u) {                           // a cell with several lists
            atomicAdd(b + 0, acc.x); atomicAdd(b + 1, acc.y);
            atomicAdd(b + 2, acc.z); atomicAdd(b + 3, acc.w);
        } else {
            float4 o = *reinterpret_cast<float4 *>(b);
            o.x += acc.x; o.y += acc.y; o.z += acc.z; o.w += acc.w;
            *reinterpret_cast<float4 *>(b) = o;
        }
    }
}

}  // namespace fda_list

#endif
