// Internal interface of the weight-gradient kernel of the per-node model (grad_tc.cu).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace retexo {

// C = A^T B reduced over `rows` batch rows, and its bias row 1^T B: A [rows x lda] holds M columns, B [rows x ldb] N.
struct GradProduct {
    const __nv_bfloat16* A; int64_t lda;
    const __nv_bfloat16* B; int64_t ldb;
    int32_t M, N;
    int32_t splits;            // ranges the rows are cut into
    float* partial;            // [splits x M x N] raw sums
    float* bias_partial;       // [splits x grad_bias_shares(M) x N] raw sums of the bias row
};

// Blocks a range's bias row is summed by.
int32_t grad_bias_shares(int32_t M);

// How the rows of one or two products (N2 = 0: one) are cut: about equal bytes per block, one block per SM.
void grad_splits(int32_t M1, int32_t N1, int32_t M2, int32_t N2, int64_t rows, int64_t* s1, int64_t* s2);

// One launch for both products of an iteration (n_products 1 or 2; the second's N is at most 64).
int grad_launch(const GradProduct* products, int n_products, int64_t rows, int32_t* status, cudaStream_t st);

}  // namespace retexo
