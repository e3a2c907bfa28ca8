// Internal interface of the GAT aggregation (gat.cu).
#pragma once
#include "common.cuh"

namespace retexo {

constexpr int kGatMaxHeads = 8;

struct GatForward {
    retexo_csr g;
    const float* p; int64_t ldp;             // projected rows
    retexo_gat_params gat;
    float* out; int64_t ldout;               // either may be null
    __nv_bfloat16* out16; int64_t ldout16;
};

void gat_forward_workspace(int64_t n_nodes, int32_t heads, Sizer& s);
// Arguments as checked by retexo_aggregate; scratch is taken from ws in the order gat_forward_workspace lists.
int gat_forward_launch(const GatForward& f, Arena& ws, int n_sm, cudaStream_t st);

}  // namespace retexo
