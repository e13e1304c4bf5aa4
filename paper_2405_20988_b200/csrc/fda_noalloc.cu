// fda_local_state_linear_noalloc: the sketch-free local state for callers that may not
// allocate.  The streaming kernel of fda_local_state (fda_rows.cuh), but the per-block partial
// sums live in a fixed array that is part of the library image, so the
// call needs no context and never calls cudaMalloc / cudaFree.
#include <mutex>

#include "fda_rows.cuh"

#define FDA_NOALLOC_MAX_BLOCKS 1024

namespace {

// Partial sums of the blocks.  Lives on every device that loads the library, until exit
// (FDA_NOALLOC_MAX_BLOCKS * FDA_NOALLOC_MAX_WORKERS * 16 bytes = 1 MiB).  In host code this
// name is only a handle for cudaGetSymbolAddress, never a device pointer.
static __device__ __align__(256) double g_noalloc_partials[FDA_NOALLOC_MAX_BLOCKS * FDA_NOALLOC_MAX_WORKERS * 2];

// The row groups' states from the partial sums, one block per group.  A second launch and not the
// last block of the first one: the ticket that would tell the last block has to be 0 when a call
// begins, and calls that overlap on the shared scratch could leave it at something else for good.
__global__ void __launch_bounds__(fda_rows::kThreads) k_noalloc_finalize(const fda_rows::Params p)
{
    __shared__ double red[fda_rows::kThreads];
    fda_grid_wait();
    fda_rows::finish_group(p, (int)blockIdx.x, red);
}

struct DeviceSetup {
    bool ready = false;
    double *partials = nullptr;     // device address of g_noalloc_partials on this device
    int n_sm = 0;
};
constexpr int kMaxDevices = 64;
DeviceSetup g_setup[kMaxDevices];
std::mutex g_setup_mutex;

}  // namespace

extern "C" fda_status fda_local_state_linear_noalloc(int device, const float *w, int64_t row_stride, int K,
                                                     int64_t d, const float *w_t0, const float *xi,
                                                     uint32_t flags, float *states, void *stream)
{
    if (!w || !w_t0 || !states) return FDA_ERR_INVALID_ARG;
    if (K < 1 || d < 1 || row_stride < d || device < 0 || device >= kMaxDevices) return FDA_ERR_INVALID_ARG;
    if (flags & ~(uint32_t)(FDA_STATE_NORM | FDA_STATE_LINEAR)) return FDA_ERR_INVALID_ARG;
    if (K > FDA_NOALLOC_MAX_WORKERS) return FDA_ERR_UNSUPPORTED;      // beyond the fixed scratch

    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess) { cudaGetLastError(); return FDA_ERR_CUDA; }
    if (device >= ndev) return FDA_ERR_INVALID_ARG;                   // no such device
    int prev = -1;
    if (cudaGetDevice(&prev) != cudaSuccess) return FDA_ERR_CUDA;
    if (prev != device && cudaSetDevice(device) != cudaSuccess) { cudaGetLastError(); return FDA_ERR_CUDA; }
    fda_status st = FDA_OK;
    DeviceSetup setup;
    {
        // first call on this device: resolve the device address of the scratch array (the
        // device is current here); no memory is allocated by this
        std::lock_guard<std::mutex> lock(g_setup_mutex);
        DeviceSetup &slot = g_setup[device];
        if (!slot.ready) {
            void *ptr = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_partials);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&slot.n_sm, cudaDevAttrMultiProcessorCount, device);
            if (e != cudaSuccess || ptr == nullptr) { cudaGetLastError(); st = FDA_ERR_CUDA; }
            else { slot.partials = static_cast<double *>(ptr); slot.ready = true; }
        }
        setup = slot;
    }
    if (st == FDA_OK) {
        fda_rows::Params p{};
        p.w = w; p.w_t0 = w_t0; p.xi = (flags & FDA_STATE_LINEAR) ? xi : nullptr;
        p.row_stride = row_stride; p.d = d; p.K = K;
        p.groups = (K + fda_rows::kRows - 1) / fda_rows::kRows;
        p.cpg = fda_rows::blocks_per_group(setup.n_sm, p.groups, d);
        p.slen = 2;
        p.flags = flags;
        p.part = setup.partials; p.states = states;
        if (p.groups * p.cpg > FDA_NOALLOC_MAX_BLOCKS) p.cpg = FDA_NOALLOC_MAX_BLOCKS / p.groups;
        cudaStream_t s = (cudaStream_t)stream;
        cudaError_t e = fda_launch_dependent(fda_rows::kernel_for<false>(p), p.groups * p.cpg, fda_rows::kThreads, 0, s, p);
        if (e == cudaSuccess) e = fda_launch_dependent(k_noalloc_finalize, p.groups, fda_rows::kThreads, 0, s, p);
        if (e != cudaSuccess) st = FDA_ERR_CUDA;
    }
    if (prev != device) cudaSetDevice(prev);
    return st;
}
