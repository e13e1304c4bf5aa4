// Local-state pass without the sketch: ||u^(k)||^2 and <xi,u^(k)> only (Section 3, local
// state; Section 3.2, LinearFDA).  The kernel is in fda_rows.cuh; here the block that finishes a
// row group last also adds the group's partial sums, so the pass is one launch.
#include "fda_rows.cuh"

// Returns cudaErrorNotSupported when a sketch is asked for.
cudaError_t fda_launch_local_state_linear(fda_ctx *ctx, const float *w, int64_t row_stride, int K,
                                          int64_t d, const float *w_t0, const float *xi,
                                          uint32_t flags, float *states, cudaStream_t s)
{
    if (flags & FDA_STATE_SKETCH) return cudaErrorNotSupported;
    fda_rows::Params p{};
    p.w = w; p.w_t0 = w_t0; p.xi = (flags & FDA_STATE_LINEAR) ? xi : nullptr;
    p.row_stride = row_stride; p.d = d; p.K = K;
    p.groups = (K + fda_rows::kRows - 1) / fda_rows::kRows;
    p.cpg = fda_rows::blocks_per_group(ctx->n_sm, p.groups, d);
    p.slen = 2 + ctx->lm;
    p.flags = flags;
    p.part = ctx->part_np; p.ticket = ctx->row_tickets; p.states = states;
    const int blocks = p.groups * p.cpg;
    if ((size_t)blocks * fda_rows::kVals > ctx->part_np_doubles) return cudaErrorNotSupported;
    return fda_launch_dependent(fda_rows::kernel_for<true>(p), blocks, fda_rows::kThreads, 0, s, p);
}
