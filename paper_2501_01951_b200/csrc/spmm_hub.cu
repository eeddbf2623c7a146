// The gather kernels over what the tiles of a graph's dense corner leave of its matrix (see hub_tiles.cu, spmm_kernels.cuh): no sampled
// aggregations, whose masks skip gathers, and no calls for the first rows only come here.  (The general group kernel keeps its test for the
// former: without it three instances spill a register.)
#define MIXGCN_SPMM_HUB 1
#include "spmm_kernels.cuh"

namespace mixgcn {

mixgcn_status launch_rows_hub(mixgcn_ctx* ctx, const SpmmHubParams& p, const SpmmSchedule& S, NarrowCfg narrow, bool loss, int phase, float* partial, cudaStream_t s) {
    return launch_rows(ctx, p, S, narrow, loss, -1, phase, partial, s);
}

}  // namespace mixgcn
