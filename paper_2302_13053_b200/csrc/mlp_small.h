// Internal interface of the two kernels that make up a training iteration of a small batch (mlp_small.cu).
#pragma once
#include "gemm_tc.h"

namespace retexo {

struct UpdateArgs;

struct SmallForward {
    const __nv_bfloat16* x; int64_t ldx;
    const __nv_bfloat16* w1t; int64_t ld_w1t;       // W1^T [out1 x ld_w1t]
    const float* b1;
    const __nv_bfloat16* w2t; int64_t ld_w2t;       // W2^T [n_classes x ld_w2t]   (hidden > 0)
    const float* b2;
    int32_t d_in, hidden, n_classes;                // hidden = 0: the first product's columns are the classes
    int64_t n_train, n_all;                         // rows [n_train, n_all) are only evaluated
    const int32_t* y; const int32_t* y_eval;
    float inv_rows;
    __nv_bfloat16* hd; int64_t ld_hd;               // Hd  [n_train x ld_hd]
    __nv_bfloat16* dl; int64_t ld_dl;               // dL  [n_train x 64]
    __nv_bfloat16* dhd; int64_t ld_dhd;             // dHd [n_train x ld_dhd]
    float* loss_partial;                            // one per 32 rows
    unsigned long long* correct;
    int32_t* status;
    bool x_early;                                   // no kernel the launch may overlap writes x
};

// Whether a training iteration of this shape takes the two kernels.
bool small_step_supported(int32_t d_in, int32_t hidden, int32_t n_classes, int64_t n_train, int64_t n_all);
int small_forward_launch(const SmallForward& f, cudaStream_t st);

// [dW1 ; db1] = [X | 1]^T grad1 and (hidden > 0) [dW2 ; db2] = [Hd | 1]^T dL, and the update `u` describes (its partials aside).
struct SmallGrad {
    const __nv_bfloat16* x; int64_t ldx;
    const __nv_bfloat16* grad1; int64_t ld_grad1;
    const __nv_bfloat16* hd; int64_t ld_hd;
    const __nv_bfloat16* dl; int64_t ld_dl;
    int64_t n_train;
    bool x_early;
};
int small_update_launch(const SmallGrad& s, const UpdateArgs& u, cudaStream_t st);

}  // namespace retexo
