#include "fda_worker_kernel.cuh"

cudaError_t fda_lanes_23(const fda_list::ListParams &p, int blocks, bool dependent, cudaStream_t s)
{
    return launch_lanes<9, 23, false, 2, 7>(p, blocks, dependent, s);
}
