#include "fda_worker_kernel.cuh"

cudaError_t fda_lanes_22(const fda_list::ListParams &p, int blocks, bool dependent, cudaStream_t s)
{
    return launch_lanes<10, 22, true, 4, 7>(p, blocks, dependent, s);
}
