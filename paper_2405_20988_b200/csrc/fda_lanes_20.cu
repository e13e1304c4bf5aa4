#include "fda_worker_kernel.cuh"

cudaError_t fda_lanes_20(const fda_list::ListParams &p, int blocks, bool dependent, cudaStream_t s)
{
    return launch_lanes<12, 20, false, 1, 7>(p, blocks, dependent, s);
}
