// cvx_surrogate.h -- internal interface of the surrogate proposal network
// (not part of the C ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "cvx_mlp.h"

struct cvx_handle;

namespace cvx {

// Flat FP32 parameters: W0 (256 x 6), b0, W1..W3 (256 x 256), b1..b3,
// W4 (7 x 256), b4 (7); weights row-major as (out, in).
constexpr long long kSurParams = 200967;

// Weights, optimiser state and batch buffers of the network (one per handle).
struct Surrogate {
    bool has_weights = false;
    float scale_h[12];  // mean (6), 1/std (6)
    float *scale = nullptr;
    float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
    __nv_bfloat16 *Wb[5] = {}, *Wt[5] = {};  // packed weights (MlpForward::W, MlpTrain::Wt)
    long long adam_t = 0;
    int rows_cap = 0;  // rows of X and out (surrogate_propose)
    __nv_bfloat16 *X = nullptr;
    float *out = nullptr;
    int cap = 0;  // rows of the training buffers (MlpTrain)
    __nv_bfloat16 *XT = nullptr, *dZoT = nullptr, *AT[4] = {}, *dZT[4] = {};
    float *Z[4] = {}, *loss = nullptr;
    int *err = nullptr;
    int *idx = nullptr;
    long long idx_cap = 0;
};

void destroy_surrogate(cvx_handle *h);
int sur_params(cvx_handle *h);
// Input and output rows of surrogate_propose's nodes, at least n.
int sur_rows(cvx_handle *h, int n);
int sur_infer(cvx_handle *h, int n, const float *X, float *out, cudaStream_t s, const int *M_dev,
              int m_off);

}  // namespace cvx
