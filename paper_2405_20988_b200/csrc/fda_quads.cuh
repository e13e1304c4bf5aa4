// Quads of four consecutive floats at any alignment, for the passes that combine the K rows of w index
// by index (fda_average.cu, fda_mean_state.cu; fda_rows.cuh, which cuts every row at its own
// boundaries, takes the helpers).  The pass runs in the frame of one vector (w_t0, or the
// averaged drifts): quad q covers indices c0 + 4q .. + 3, where that vector is 16-byte aligned.  A row
// aligned otherwise is read as the two aligned quads around those indices, with 128-bit loads of which
// the second hits L1, and written as quads at its own boundaries, put together from two neighbouring lanes.
#ifndef FDA_QUADS_CUH_
#define FDA_QUADS_CUH_

#include <cuda_runtime.h>
#include <stdint.h>

namespace fda_quads {

// distance of a pointer from the 16-byte boundary below it, in floats
__host__ __device__ __forceinline__ int misaligned(const float *ptr) { return (int)(((uintptr_t)ptr >> 2) & 3u); }
// first index at which the vector is aligned
__host__ __device__ __forceinline__ int first_aligned(const float *ptr) { return (4 - misaligned(ptr)) & 3; }

// four of the eight values a, b from position r on
__device__ __forceinline__ float4 pick(const float4 &a, const float4 &b, int r)
{
    switch (r) {
        case 0: return a;
        case 1: return make_float4(a.y, a.z, a.w, b.x);
        case 2: return make_float4(a.z, a.w, b.x, b.y);
        default: return make_float4(a.w, b.x, b.y, b.z);
    }
}

// The two aligned quads around ptr .. ptr + 3 (one when ptr is aligned).  Reads up to three floats in
// front of ptr and four behind ptr + 3: the caller keeps away from the ends of the row.
struct Window {
    float4 a, b;
};
__device__ __forceinline__ Window load_window(const float *ptr)
{
    const float4 *q = reinterpret_cast<const float4 *>((uintptr_t)ptr & ~(uintptr_t)15);
    Window w;
    w.a = q[0];
    w.b = q[misaligned(ptr) ? 1 : 0];
    return w;
}
__device__ __forceinline__ float4 value(const Window &w, const float *ptr) { return pick(w.a, w.b, misaligned(ptr)); }

// Stores v at ptr .. ptr + 3 when the lanes of a warp hold consecutive quads: ptr is lane 0's pointer + 4
// * lane, nx the first three values of the next lane.  The quad that starts at the row's boundary
// inside this lane's four goes out as one store; what has no whole quad at the ends of the warp's
// run as single floats.
__device__ __forceinline__ void store_shifted(float *ptr, const float4 &v, const float4 &nx, bool first, bool last)
{
    const int r = (4 - misaligned(ptr)) & 3;              // floats in front of the boundary
    if (!last || r == 0) __stcs(reinterpret_cast<float4 *>(ptr + r), pick(v, nx, r));
    else {
        if (r < 2) __stcs(ptr + 1, v.y);
        if (r < 3) __stcs(ptr + 2, v.z);
        __stcs(ptr + 3, v.w);
    }
    if (first && r > 0) {
        __stcs(ptr, v.x);
        if (r > 1) __stcs(ptr + 1, v.y);
        if (r > 2) __stcs(ptr + 2, v.z);
    }
}

}  // namespace fda_quads

#endif
