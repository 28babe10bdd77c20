// cvx_mlp.h -- internal interface of the surrogate network's tensor-core
// kernels (not part of the C ABI).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace cvx {

// The result of launch_gemm: C (M_valid x N, FP32).
struct GemmEpi {
    int M_valid;
    float *C;
    int ldc;
    int *err;  // set to 1 if a wait timed out
};

// 2-D tensor map of a row-major bf16 matrix (rows x cols, leading dimension ld
// elements) read in boxes of 8 columns x box_rows rows.  false if the CUDA
// driver's entry point is missing or the layout breaks the TMA rules.
bool make_tmap_bf16(CUtensorMap *map, const void *ptr, long long rows, long long cols,
                    long long ld, int box_rows);

// C = A B^T over M x N (tiles of 128 x BN, BN = 16 or 256), K a multiple of
// 16.  tA: box rows 128; tB: box rows BN.
cudaError_t launch_gemm(const CUtensorMap &tA, const CUtensorMap &tB, int M, int N, int K,
                        int BN, const GemmEpi &ep, cudaStream_t s);

// Inference of the whole network in one kernel (cvx_mlp_fused.cu).
struct MlpForward {
    int M;             // rows
    const int *M_dev;  // optional device-side row count; rows valid = *M_dev - m_off
    int m_off;
    const float *X;            // M x 6 raw features, standardised with scale, or
    const __nv_bfloat16 *X16;  // M x 16 standardised rows (X unused)
    const float *scale;        // mean (6), 1 / deviation (6)
    // weights as k-blocks of 8 elements x all output rows (256, or 16 for the
    // last layer) x 16 bytes
    const __nv_bfloat16 *W[5];
    const float *bias[5];
    float *out;  // M x 7
    int *err;    // set to 1 if a wait timed out
};
cudaError_t launch_mlp_forward(const MlpForward &f, cudaStream_t s);

// Mean loss and its gradient over n rows (cvx_mlp_train.cu), added to loss,
// dbias and dW.
struct MlpTrain {
    int n;
    long long ld;     // rows of the buffers below, a multiple of 128
    const int *idx;   // optional: row m is sample idx[m]
    const float *X;   // x 6 raw features, standardised with scale
    const float *Y;   // x 7 labels
    const float *scale;
    const __nv_bfloat16 *W[5];   // as MlpForward::W
    const __nv_bfloat16 *Wt[5];  // transposed weights of layers 1-4 in the same layout
    const float *bias[5];
    // per hidden layer: Z (FP32, [column / 4][row][4]); A and dZ (BF16) with
    // element (row, column) at ((row / 8) width + column) 8 + row % 8, as the
    // input XT (width 16) and the output gradient dZoT (width 16)
    float *Z[4];
    __nv_bfloat16 *AT[4], *dZT[4], *XT, *dZoT;
    float *dW[5], *dbias[5];  // gradients, weights row-major (out, in)
    float *loss;
    int *err;  // set to 1 if a wait timed out
};
cudaError_t launch_mlp_grad(const MlpTrain &f, cudaStream_t s);

}  // namespace cvx
