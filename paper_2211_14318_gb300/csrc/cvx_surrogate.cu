// cvx_surrogate.cu -- the surrogate proposal network: parameters, BF16
// packing, Adam, training, save/load.  Inference is one kernel
// (cvx_mlp_fused.cu), the loss and its gradient are two (cvx_mlp_train.cu).
//
// Network: x = standardised (F11, F12, F21, F22, beta_k, ln det F) ->
// 4 x [256, GELU] -> 7 outputs (two direction angles, the logit of the volume
// fraction, the four entries of the jump F+ - F-).  Weights are kept in FP32
// (master copy, Adam state) and packed to BF16 for the tensor cores, in both
// orientations (W for the forward pass, W^T for back-propagation).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <random>
#include <vector>

#include "cvx_handle.h"
#include "cvx_mlp.h"
#include "cvx_surrogate.h"

namespace cvx {

namespace {

constexpr long long kWOff[5] = {0, 1792, 67584, 133376, 199168};
constexpr long long kBOff[5] = {1536, 67328, 133120, 198912, 200960};
constexpr int kOut[5] = {256, 256, 256, 256, 7};
constexpr int kIn[5] = {6, 256, 256, 256, 256};
static_assert(kBOff[4] + 7 == kSurParams, "parameter layout");

using bf16 = __nv_bfloat16;

// ------------------------------------------------------------------ kernels
struct Packed {
    bf16 *W[5], *Wt[5];
};

// Parameter i, if it is a weight, to its places in the packed operands: W[r][c]
// of layer l as k-blocks of 8 columns x all rows (256; 16 for the last layer)
// and W^T likewise (layers 1-4).  The padding stays zero.
__device__ __forceinline__ void pack_weight(long long i, float w, const Packed &p) {
#pragma unroll
    for (int l = 0; l < 5; ++l) {
        const int in = l ? 256 : 6, out = l < 4 ? 256 : 7;
        constexpr long long kOff[5] = {0, 1792, 67584, 133376, 199168};  // kWOff
        const long long k = i - kOff[l];
        if (k < 0 || k >= (long long)in * out) continue;
        const int r = (int)(k / in), c = (int)(k % in);
        const bf16 b = __float2bfloat16_rn(w);
        p.W[l][((c >> 3) * (l < 4 ? 256 : 16) + r) * 8 + (c & 7)] = b;
        if (l) p.Wt[l][((r >> 3) * 256 + c) * 8 + (r & 7)] = b;
    }
}

__global__ void k_pack(long long n, const float *w, Packed p) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) pack_weight(i, w[i], p);
}

// One Adam step, and the packed weights of the result.
__global__ void k_adam(long long n, float *w, const float *g, float *m, float *v, float lr,
                       float b1, float b2, float eps, float c1, float c2, Packed p) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    pack_weight(i, wi, p);
}

template <typename T>
cudaError_t alloc(T **p, size_t count) {
    return cudaMalloc(reinterpret_cast<void **>(p), sizeof(T) * count);
}

}  // namespace

void destroy_surrogate(cvx_handle *h) {
    Surrogate *S = h->sur;
    if (!S) return;
    void *ptrs[] = {S->scale, S->w, S->g, S->m, S->v, S->X, S->out, S->XT, S->dZoT, S->loss, S->err,
                    S->idx};
    for (void *p : ptrs) cudaFree(p);
    for (int l = 0; l < 5; ++l) {
        cudaFree(S->Wb[l]);
        cudaFree(S->Wt[l]);
    }
    for (int l = 0; l < 4; ++l) {
        cudaFree(S->AT[l]);
        cudaFree(S->dZT[l]);
        cudaFree(S->Z[l]);
    }
    delete S;
    h->sur = nullptr;
}

int sur_params(cvx_handle *h) {
    if (h->sur && h->sur->w) return CVX_OK;
    if (!h->sur) h->sur = new Surrogate();
    Surrogate &S = *h->sur;
    CK(alloc(&S.scale, 12), "surrogate");
    CK(alloc(&S.w, kSurParams), "surrogate");
    CK(alloc(&S.g, kSurParams), "surrogate");
    CK(alloc(&S.m, kSurParams), "surrogate");
    CK(alloc(&S.v, kSurParams), "surrogate");
    CK(alloc(&S.loss, 1), "surrogate");
    CK(alloc(&S.err, 1), "surrogate");
    CK(cudaMemset(S.err, 0, sizeof(int)), "surrogate");
    for (int l = 0; l < 5; ++l) {
        const size_t n = l == 0 || l == 4 ? 256 * 16 : 256 * 256;
        CK(alloc(&S.Wb[l], n), "surrogate");
        CK(cudaMemset(S.Wb[l], 0, sizeof(bf16) * n), "surrogate");
        CK(alloc(&S.Wt[l], n), "surrogate");
        CK(cudaMemset(S.Wt[l], 0, sizeof(bf16) * n), "surrogate");
    }
    // the handle's calls may use any stream, which the legacy stream's fills do
    // not precede by themselves
    CK(cudaDeviceSynchronize(), "surrogate");
    return CVX_OK;
}

int sur_rows(cvx_handle *h, int n) {
    Surrogate &S = *h->sur;
    if (n <= S.rows_cap) return CVX_OK;
    const size_t cap = (size_t)((n + 127) / 128) * 128;
    cudaDeviceSynchronize();
    cudaFree(S.X);
    cudaFree(S.out);
    S.X = nullptr;
    S.out = nullptr;
    S.rows_cap = 0;
    CK(alloc(&S.X, cap * 16), "surrogate rows");
    CK(alloc(&S.out, cap * 7), "surrogate rows");
    S.rows_cap = (int)cap;
    return CVX_OK;
}

namespace {

// Training buffers for at least n rows.
int sur_batch(cvx_handle *h, int n) {
    Surrogate &S = *h->sur;
    if (n <= S.cap) return CVX_OK;
    const size_t cap = (size_t)((n + 127) / 128) * 128;
    cudaDeviceSynchronize();
    cudaFree(S.XT);
    cudaFree(S.dZoT);
    S.XT = S.dZoT = nullptr;
    for (int l = 0; l < 4; ++l) {
        cudaFree(S.AT[l]);
        cudaFree(S.dZT[l]);
        cudaFree(S.Z[l]);
        S.AT[l] = S.dZT[l] = nullptr;
        S.Z[l] = nullptr;
    }
    S.cap = 0;
    CK(alloc(&S.XT, cap * 16), "surrogate batch");
    CK(alloc(&S.dZoT, cap * 16), "surrogate batch");
    for (int l = 0; l < 4; ++l) {
        CK(alloc(&S.AT[l], cap * 256), "surrogate batch");
        CK(alloc(&S.dZT[l], cap * 256), "surrogate batch");
        CK(alloc(&S.Z[l], cap * 256), "surrogate batch");
    }
    S.cap = (int)cap;
    return CVX_OK;
}

Packed packed(const Surrogate &S) {
    Packed p;
    for (int l = 0; l < 5; ++l) {
        p.W[l] = S.Wb[l];
        p.Wt[l] = S.Wt[l];
    }
    return p;
}

cudaError_t sur_pack(Surrogate &S, cudaStream_t s) {
    k_pack<<<(kSurParams + 255) / 256, 256, 0, s>>>(kSurParams, S.w, packed(S));
    return cudaGetLastError();
}

}  // namespace

// Inference of n rows in one kernel: raw features X, or (X null) the
// standardised rows in S.X.  M_dev (optional): device-side row count, of which
// rows m_off .. m_off + n - 1 are these.
int sur_infer(cvx_handle *h, int n, const float *X, float *out, cudaStream_t s, const int *M_dev,
              int m_off) {
    Surrogate &S = *h->sur;
    MlpForward f = {};
    f.M = n;
    f.M_dev = M_dev;
    f.m_off = m_off;
    f.X = X;
    f.X16 = X ? nullptr : S.X;
    f.scale = S.scale;
    for (int l = 0; l < 5; ++l) {
        f.W[l] = S.Wb[l];
        f.bias[l] = S.w + kBOff[l];
    }
    f.out = out;
    f.err = S.err;
    CK(launch_mlp_forward(f, s), "surrogate forward");
    return CVX_OK;
}

namespace {

// Loss and gradient (added to loss and g, 16-byte aligned) of n <= cap samples,
// row m being sample idx[m] (or m).
int sur_grad(cvx_handle *h, int n, const int *idx, const float *X, const float *Y, float *loss,
             float *g, cudaStream_t s) {
    Surrogate &S = *h->sur;
    MlpTrain f = {};
    f.n = n;
    f.ld = S.cap;
    f.idx = idx;
    f.X = X;
    f.Y = Y;
    f.scale = S.scale;
    for (int l = 0; l < 5; ++l) {
        f.W[l] = S.Wb[l];
        f.Wt[l] = S.Wt[l];
        f.bias[l] = S.w + kBOff[l];
        f.dW[l] = g + kWOff[l];
        f.dbias[l] = g + kBOff[l];
    }
    for (int l = 0; l < 4; ++l) {
        f.Z[l] = S.Z[l];
        f.AT[l] = S.AT[l];
        f.dZT[l] = S.dZT[l];
    }
    f.XT = S.XT;
    f.dZoT = S.dZoT;
    f.loss = loss;
    f.err = S.err;
    CK(launch_mlp_grad(f, s), "surrogate gradient");
    return CVX_OK;
}

int check_err(Surrogate &S, cudaStream_t s) {
    int e = 0;
    CK(cudaMemcpyAsync(&e, S.err, sizeof(int), cudaMemcpyDeviceToHost, s), "surrogate");
    CK(cudaStreamSynchronize(s), "surrogate");
    if (e) {
        cudaMemsetAsync(S.err, 0, sizeof(int), s);
        return fail(CVX_ERR_TIMEOUT, "a tensor-core pipeline wait timed out");
    }
    return CVX_OK;
}

void init_host(std::vector<float> &p, uint64_t seed) {
    std::mt19937_64 rng(seed);
    p.assign(kSurParams, 0.0f);
    for (int l = 0; l < 5; ++l) {
        const float b = 1.0f / sqrtf((float)kIn[l]);
        std::uniform_real_distribution<float> u(-b, b);
        for (long long i = 0; i < (long long)kOut[l] * kIn[l]; ++i) p[kWOff[l] + i] = u(rng);
        for (int i = 0; i < kOut[l]; ++i) p[kBOff[l] + i] = u(rng);
    }
}

int upload_weights(cvx_handle *h, const float *params, const float *mean, const float *stdv,
                   cudaStream_t s) {
    Surrogate &S = *h->sur;
    for (int k = 0; k < 6; ++k) {
        if (!(stdv[k] > 0.0f) || !isfinite(mean[k]))
            return fail(CVX_ERR_INVALID_ARG, "input scaling: std must be > 0");
        S.scale_h[k] = mean[k];
        S.scale_h[6 + k] = 1.0f / stdv[k];
    }
    // on the stream that reads them next (pageable sources: staged at return)
    CK(cudaMemcpyAsync(S.scale, S.scale_h, sizeof(float) * 12, cudaMemcpyHostToDevice, s), "surrogate");
    CK(cudaMemcpyAsync(S.w, params, sizeof(float) * kSurParams, cudaMemcpyHostToDevice, s), "surrogate");
    CK(cudaMemsetAsync(S.m, 0, sizeof(float) * kSurParams, s), "surrogate");
    CK(cudaMemsetAsync(S.v, 0, sizeof(float) * kSurParams, s), "surrogate");
    S.adam_t = 0;
    CK(sur_pack(S, s), "surrogate pack");
    S.has_weights = true;
    return CVX_OK;
}

}  // namespace

}  // namespace cvx

using namespace cvx;

extern "C" {

int cvx_gemm_bf16(cvx_handle *h, int M, int N, int K, const uint16_t *A, const uint16_t *B,
                  float *C, cvx_stream sv) {
    if (!h) return fail(CVX_ERR_INVALID_ARG, "handle is NULL");
    if (M < 1 || N < 1 || K < 16 || K % 16) return fail(CVX_ERR_INVALID_ARG, "need M, N >= 1 and K a positive multiple of 16");
    if (!A || !B || !C) return fail(CVX_ERR_INVALID_ARG, "NULL array");
    DeviceGuard g(h->device);
    CUtensorMap ta, tb;
    const int BN = N <= 16 ? 16 : 256;
    if (!make_tmap_bf16(&ta, A, M, K, K, 128) || !make_tmap_bf16(&tb, B, N, K, K, BN))
        return fail(CVX_ERR_CUDA, "cvx_gemm_bf16: tensor map failed");
    int rc = sur_params(h);
    if (rc) return rc;
    GemmEpi e = {};
    e.M_valid = M;
    e.err = h->sur->err;
    e.C = C;
    e.ldc = N;
    CK(launch_gemm(ta, tb, M, N, K, BN, e, (cudaStream_t)sv), "cvx_gemm_bf16");
    return check_err(*h->sur, (cudaStream_t)sv);
}

int surrogate_set_weights(cvx_handle *h, const float *params, const float *mean,
                          const float *stdv) {
    if (!h || !params || !mean || !stdv) return fail(CVX_ERR_INVALID_ARG, "NULL argument");
    DeviceGuard g(h->device);
    int rc = sur_params(h);
    if (rc) return rc;
    rc = upload_weights(h, params, mean, stdv, 0);
    if (rc) return rc;
    CK(cudaDeviceSynchronize(), "surrogate_set_weights");
    return CVX_OK;
}

int surrogate_get_weights(cvx_handle *h, float *params, float *mean, float *stdv) {
    if (!h || !params || !mean || !stdv) return fail(CVX_ERR_INVALID_ARG, "NULL argument");
    if (!h->sur || !h->sur->has_weights) return fail(CVX_ERR_NOT_TRAINED, "no surrogate weights");
    DeviceGuard g(h->device);
    Surrogate &S = *h->sur;
    CK(cudaDeviceSynchronize(), "surrogate_get_weights");
    CK(cudaMemcpy(params, S.w, sizeof(float) * kSurParams, cudaMemcpyDeviceToHost), "surrogate_get_weights");
    for (int k = 0; k < 6; ++k) {
        mean[k] = S.scale_h[k];
        stdv[k] = 1.0f / S.scale_h[6 + k];
    }
    return CVX_OK;
}

int surrogate_forward(cvx_handle *h, int64_t n, const float *X, float *out, cvx_stream sv) {
    if (!h) return fail(CVX_ERR_INVALID_ARG, "handle is NULL");
    if (n < 0) return fail(CVX_ERR_INVALID_ARG, "n < 0");
    if (n > 0 && (!X || !out)) return fail(CVX_ERR_INVALID_ARG, "NULL array");
    if (!h->sur || !h->sur->has_weights) return fail(CVX_ERR_NOT_TRAINED, "no surrogate weights");
    if (n == 0) return CVX_OK;
    DeviceGuard g(h->device);
    cudaStream_t s = (cudaStream_t)sv;
    Surrogate &S = *h->sur;
    const int64_t chunk = (int64_t)1 << 30;  // rows per launch
    for (int64_t o = 0; o < n; o += chunk) {
        const int rc = sur_infer(h, (int)std::min<int64_t>(chunk, n - o), X + 6 * o, out + 7 * o, s,
                                 nullptr, 0);
        if (rc) return rc;
    }
    return check_err(S, s);
}

int surrogate_loss_grad(cvx_handle *h, int64_t n, const float *X, const float *Y, float *loss,
                        float *grad, cvx_stream sv) {
    if (!h) return fail(CVX_ERR_INVALID_ARG, "handle is NULL");
    if (n < 1 || n > (1 << 20)) return fail(CVX_ERR_INVALID_ARG, "n must be in [1, 2^20]");
    if (!X || !Y || !loss || !grad) return fail(CVX_ERR_INVALID_ARG, "NULL array");
    if (!h->sur || !h->sur->has_weights) return fail(CVX_ERR_NOT_TRAINED, "no surrogate weights");
    DeviceGuard g(h->device);
    cudaStream_t s = (cudaStream_t)sv;
    Surrogate &S = *h->sur;
    int rc = sur_batch(h, (int)n);
    if (rc) return rc;
    // straight into the caller's gradient where its alignment allows the paired
    // additions
    float *g_out = ((uintptr_t)grad & 15) == 0 ? grad : S.g;
    CK(cudaMemsetAsync(g_out, 0, sizeof(float) * kSurParams, s), "surrogate_loss_grad");
    CK(cudaMemsetAsync(loss, 0, sizeof(float), s), "surrogate_loss_grad");
    rc = sur_grad(h, (int)n, nullptr, X, Y, loss, g_out, s);
    if (rc) return rc;
    if (g_out != grad)
        CK(cudaMemcpyAsync(grad, S.g, sizeof(float) * kSurParams, cudaMemcpyDeviceToDevice, s), "surrogate_loss_grad");
    return check_err(S, s);
}

int surrogate_train(cvx_handle *h, int64_t n, const float *X, const float *Y,
                    const cvx_train_cfg *cfg, float *loss_log, cvx_stream sv) {
    if (!h || !cfg) return fail(CVX_ERR_INVALID_ARG, "NULL argument");
    if (n < 1 || n > ((int64_t)1 << 31) - 1) return fail(CVX_ERR_INVALID_ARG, "n out of range");
    if (!X || !Y) return fail(CVX_ERR_INVALID_ARG, "NULL array");
    if (cfg->epochs < 0 || cfg->batch < 16 || cfg->batch > (1 << 16) || !(cfg->lr > 0.0f))
        return fail(CVX_ERR_INVALID_ARG, "train cfg: epochs >= 0, 16 <= batch <= 65536, lr > 0");
    DeviceGuard g(h->device);
    cudaStream_t s = (cudaStream_t)sv;
    int rc = sur_params(h);
    if (rc) return rc;
    Surrogate &S = *h->sur;
    if (cfg->init || !S.has_weights) {
        // input standardisation from the data, fresh weights
        std::vector<float> x((size_t)n * 6);
        CK(cudaMemcpyAsync(x.data(), X, sizeof(float) * x.size(), cudaMemcpyDeviceToHost, s), "surrogate_train");
        CK(cudaStreamSynchronize(s), "surrogate_train");
        float mean[6], stdv[6];
        for (int k = 0; k < 6; ++k) {
            double a = 0.0, b = 0.0;
            for (int64_t i = 0; i < n; ++i) a += x[(size_t)i * 6 + k];
            a /= (double)n;
            for (int64_t i = 0; i < n; ++i) b += (x[(size_t)i * 6 + k] - a) * (x[(size_t)i * 6 + k] - a);
            mean[k] = (float)a;
            stdv[k] = (float)std::max(sqrt(b / (double)n), 1e-6);
        }
        std::vector<float> p;
        init_host(p, cfg->seed);
        rc = upload_weights(h, p.data(), mean, stdv, s);
        if (rc) return rc;
    }
    const int B = cfg->batch;
    rc = sur_batch(h, B);
    if (rc) return rc;
    if (S.idx_cap < n) {
        cudaFree(S.idx);
        S.idx = nullptr;
        S.idx_cap = 0;
        CK(alloc(&S.idx, (size_t)n), "surrogate_train");
        S.idx_cap = n;
    }
    std::vector<int> perm((size_t)n);
    for (int64_t i = 0; i < n; ++i) perm[(size_t)i] = (int)i;
    std::mt19937_64 rng(cfg->seed ^ 0x9E3779B97F4A7C15ull);
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    for (int ep = 0; ep < cfg->epochs; ++ep) {
        std::shuffle(perm.begin(), perm.end(), rng);
        CK(cudaMemcpyAsync(S.idx, perm.data(), sizeof(int) * (size_t)n, cudaMemcpyHostToDevice, s), "surrogate_train");
        CK(cudaMemsetAsync(S.loss, 0, sizeof(float), s), "surrogate_train");
        int batches = 0;
        for (int64_t o = 0; o + B <= n || (o == 0 && n < B); o += B) {
            const int m = (int)std::min<int64_t>(B, n - o);
            CK(cudaMemsetAsync(S.g, 0, sizeof(float) * kSurParams, s), "surrogate_train");
            rc = sur_grad(h, m, S.idx + o, X, Y, S.loss, S.g, s);
            if (rc) return rc;
            ++S.adam_t;
            const float c1 = 1.0f - powf(b1, (float)S.adam_t), c2 = 1.0f - powf(b2, (float)S.adam_t);
            k_adam<<<(kSurParams + 255) / 256, 256, 0, s>>>(kSurParams, S.w, S.g, S.m, S.v, cfg->lr, b1, b2, eps, c1, c2, packed(S));
            CK(cudaGetLastError(), "surrogate_train");
            ++batches;
            if (n < B) break;
        }
        rc = check_err(S, s);
        if (rc) return rc;
        if (loss_log) {
            float l = 0.0f;
            CK(cudaMemcpy(&l, S.loss, sizeof(float), cudaMemcpyDeviceToHost), "surrogate_train");
            loss_log[ep] = l / (float)std::max(batches, 1);
        }
    }
    CK(cudaStreamSynchronize(s), "surrogate_train");
    return CVX_OK;
}

int surrogate_save(cvx_handle *h, const char *path) {
    if (!h || !path) return fail(CVX_ERR_INVALID_ARG, "NULL argument");
    if (!h->sur || !h->sur->has_weights) return fail(CVX_ERR_NOT_TRAINED, "no surrogate weights");
    std::vector<float> p(kSurParams);
    float mean[6], stdv[6];
    int rc = surrogate_get_weights(h, p.data(), mean, stdv);
    if (rc) return rc;
    FILE *f = fopen(path, "wb");
    if (!f) return fail(CVX_ERR_INVALID_ARG, "cannot open %s", path);
    const char magic[8] = {'C', 'V', 'X', 'S', 'U', 'R', '0', '1'};
    const int32_t np = (int32_t)kSurParams;
    bool ok = fwrite(magic, 1, 8, f) == 8 && fwrite(&np, 4, 1, f) == 1 &&
              fwrite(mean, 4, 6, f) == 6 && fwrite(stdv, 4, 6, f) == 6 &&
              fwrite(p.data(), 4, p.size(), f) == p.size();
    ok = (fclose(f) == 0) && ok;
    return ok ? CVX_OK : fail(CVX_ERR_INVALID_ARG, "write to %s failed", path);
}

int surrogate_load(cvx_handle *h, const char *path) {
    if (!h || !path) return fail(CVX_ERR_INVALID_ARG, "NULL argument");
    FILE *f = fopen(path, "rb");
    if (!f) return fail(CVX_ERR_INVALID_ARG, "cannot open %s", path);
    char magic[8];
    int32_t np = 0;
    float mean[6], stdv[6];
    std::vector<float> p(kSurParams);
    bool ok = fread(magic, 1, 8, f) == 8 && memcmp(magic, "CVXSUR01", 8) == 0 &&
              fread(&np, 4, 1, f) == 1 && np == (int32_t)kSurParams && fread(mean, 4, 6, f) == 6 &&
              fread(stdv, 4, 6, f) == 6 && fread(p.data(), 4, p.size(), f) == p.size();
    fclose(f);
    if (!ok) return fail(CVX_ERR_INVALID_ARG, "%s is not a surrogate file", path);
    return surrogate_set_weights(h, p.data(), mean, stdv);
}

}  // extern "C"
