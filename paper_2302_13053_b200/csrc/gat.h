// Internal interface of the GAT aggregation (gat.cu).
#pragma once
#include "common.cuh"

namespace retexo {

constexpr int kGatMaxHeads = 8;

struct GatRow;
// Rows of a graph in order of falling length (gat_lanes.cuh), where the caller keeps them: the lane kernels then take these rows only.
struct GatRowOrder {
    const GatRow* rows;         // null: built by the call, over all rows
    const int32_t* counts;      // (device) how many of the first rows are hubs, and how many are above kGatGroupEntries
    const int32_t* slots;       // null, or the row of the bf16 output that entry i goes to (else: its node's)
    int64_t n;                  // rows listed
};

struct GatForward {
    retexo_csr g;
    const float* p; int64_t ldp;             // projected rows
    retexo_gat_params gat;
    float* out; int64_t ldout;               // either may be null
    __nv_bfloat16* out16; int64_t ldout16;
    GatRowOrder order;
};

void gat_forward_workspace(int64_t n_nodes, int32_t heads, Sizer& s);
bool gat_lanes_usable(int32_t heads, int32_t head_dim, const float* p, int64_t ldp, const float* q, int64_t ldq);
constexpr int kGatOrderCounts = 256, kGatOrderInts = kGatOrderCounts + 64;      // rows per class of lengths, rows placed so far, GatRowOrder::counts
// Builds the order of the rows of some index lists (a null list: all rows); its counts are at bins + kGatOrderCounts.  rows, slots (optional:
// slots count on through the lists): one entry per row listed; bins: kGatOrderInts words; rows of hub_entries
// or more are hubs.
int gat_order_launch(const retexo_csr& g, int32_t self_loop, const int32_t* const* idx, const int64_t* n_idx, int lists, GatRow* rows,
                     int32_t* slots, int32_t* bins, int hub_entries, cudaStream_t st);
// Arguments as checked by retexo_aggregate; scratch is taken from ws in the order gat_forward_workspace lists.
int gat_forward_launch(const GatForward& f, Arena& ws, int n_sm, cudaStream_t st);

// The scores that pass left in its scratch ([n x heads] each), for the backward pass of the same rows.
inline const float* gat_forward_s(void* ws) { return static_cast<const float*>(ws); }
inline const float* gat_forward_t(void* ws, int64_t n, int32_t heads) {
    return reinterpret_cast<const float*>(static_cast<char*>(ws) + align_up(sizeof(float) * (size_t)n * (size_t)heads));
}

// What a caller of retexo_gat_backward that makes many passes over one graph keeps between them (lane layout only).
struct GatBackwardKept {
    GatRowOrder dst, src;       // dst: rows whose gradient may be other than zero; src: all rows, of the entries in src_colidx
    const int32_t* src_colidx;  // the graph's entries whose column is in dst
    const float* s; const float* t;
};
// Before the first pass with `kept`: clears what the passes leave as it is for rows that dst does not list.
int gat_backward_prepare(int64_t n_nodes, int64_t n_edges, int32_t heads, int32_t head_dim, void* workspace, size_t workspace_bytes, cudaStream_t st);
// retexo_gat_backward; kept: optional.
int gat_backward(const retexo_csr* g, const float* p, int64_t ldp, const retexo_gat_params* gat, const float* dz, int64_t lddz, float* dp,
                 int64_t lddp, void* dp_bf16, int64_t lddp_bf16, float* da_src, float* da_dst, void* workspace, size_t workspace_bytes,
                 const GatBackwardKept* kept, cudaStream_t st);

}  // namespace retexo
