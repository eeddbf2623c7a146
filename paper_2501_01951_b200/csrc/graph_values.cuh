// Values of a graph's matrix, for the kernels that build it.
#pragma once
#include <stdint.h>

namespace mixgcn {

// Value of an entry of row u.  norm 0: dinv_u * dinv_v (Section 2.1); 1: 1 / (entries in row u), the row mean (GraphSAGE's
// mean aggregator; IEEE reciprocal); 2: 1, the plain sum (GIN's sum aggregator).
__device__ __forceinline__ float entry_value(int norm, float dinv_u, float dinv_v, int32_t deg_u) {
    return norm == 0 ? __fmul_rn(dinv_u, dinv_v) : norm == 1 ? __frcp_rn((float)deg_u) : 1.0f;
}
// dinv = 1/sqrt(deg): IEEE square root, then IEEE reciprocal, each rounded to fp32.
__device__ __forceinline__ float degree_norm(int32_t d) { return d > 0 ? __frcp_rn(__fsqrt_rn((float)d)) : 0.0f; }

}  // namespace mixgcn
