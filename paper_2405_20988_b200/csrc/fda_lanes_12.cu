#include "fda_worker_kernel.cuh"

cudaError_t fda_lanes_12(const fda_list::ListParams &p, int blocks, bool dependent, cudaStream_t s)
{
    return launch_lanes<16, 12, false, 1, 2>(p, blocks, dependent, s);
}
