// The gather kernels over what the tiles of a graph's dense corner leave of its matrix (see hub_tiles.cu, spmm_kernels.cuh).
#define MIXGCN_SPMM_HUB 1
#include "spmm_kernels.cuh"

namespace mixgcn {

mixgcn_status launch_rows_hub(mixgcn_ctx* ctx, const SpmmHubParams& p, const SpmmSchedule& S, NarrowCfg narrow, bool loss, int64_t row_limit, int phase, float* partial, cudaStream_t s) {
    return launch_rows(ctx, p, S, narrow, loss, row_limit, phase, partial, s);
}

}  // namespace mixgcn
