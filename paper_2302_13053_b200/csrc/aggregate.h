// Internal: the aggregation call of the library's own loops.
#pragma once
#include <stddef.h>

#include "retexo.h"

namespace retexo {

// retexo_aggregate for a matrix whose memory (whole_rows) holds the last row's full stride as well, so that its ragged end may
// be read in 32-byte pieces.
int aggregate_rows(const retexo_csr* g, int32_t type, const float* q, int64_t ldq, int32_t dim, bool whole_rows,
                   const retexo_gat_params* gat, float* out, int64_t ldout, int32_t concat_self, void* out_bf16,
                   int64_t ldout_bf16, void* workspace, size_t workspace_bytes, void* stream);

}  // namespace retexo
