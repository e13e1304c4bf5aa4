#include "fda_worker_kernel.cuh"

cudaError_t fda_lanes_24(const fda_list::ListParams &p, int blocks, bool dependent, cudaStream_t s)
{
    return launch_lanes<8, 24, false, 2, 6>(p, blocks, dependent, s);
}
