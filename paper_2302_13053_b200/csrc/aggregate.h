// Internal: the aggregation calls of the library's own loops (GCN, SAGE mean and max).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include "retexo.h"

namespace retexo {

// retexo_aggregate, except that it gathers rows which are to be weighted as they are, whatever pieces they come in; whole_rows: the
// matrix's memory holds the last row's full stride as well, so that the row's ragged end may be read in 32-byte pieces.
int aggregate_rows(const retexo_csr* g, int32_t type, const float* q, int64_t ldq, int32_t dim, bool whole_rows, float* out,
                   int64_t ldout, int32_t concat_self, void* out_bf16, int64_t ldout_bf16, void* workspace, size_t workspace_bytes,
                   void* stream);

// What that call needs, or (lay_out) retexo_aggregate with any alignment.
size_t aggregate_rows_workspace_size(int64_t n_nodes, int64_t n_edges, int32_t type, int32_t dim, int32_t heads, bool lay_out);

// Whether that call reads its rows once to copy them, so that it does not matter much in what pieces they come.
bool aggregate_copies_rows(int64_t n_nodes, int64_t n_edges, int32_t type, int32_t dim);

// dst[i] = [src[i] | zeros] for n rows of dim floats: rows of ld_dst (a multiple of 4) floats from dense or strided ones.
int relay_rows_launch(const float* src, int64_t ld_src, int32_t dim, int64_t n, float* dst, int64_t ld_dst, cudaStream_t st);

}  // namespace retexo
