// Internal: the aggregation calls of the library's own loops (GCN, SAGE mean and max), whose rows come in 16-byte pieces.
#pragma once
#include <stddef.h>

#include "retexo.h"

namespace retexo {

// retexo_aggregate for such a matrix; whole_rows: its memory holds the last row's full stride as well, so that the row's ragged
// end may be read in 32-byte pieces.
int aggregate_rows(const retexo_csr* g, int32_t type, const float* q, int64_t ldq, int32_t dim, bool whole_rows, float* out,
                   int64_t ldout, int32_t concat_self, void* out_bf16, int64_t ldout_bf16, void* workspace, size_t workspace_bytes,
                   void* stream);

// What that call needs (pieces16), or retexo_aggregate with any alignment.
size_t aggregate_rows_workspace_size(int64_t n_nodes, int64_t n_edges, int32_t type, int32_t dim, int32_t heads, bool pieces16);

}  // namespace retexo
