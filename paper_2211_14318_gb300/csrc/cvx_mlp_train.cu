// cvx_mlp_train.cu -- the gradient of the surrogate network's loss over one
// batch in two kernels.
//
// k_mlp_train takes a tile of 128 rows through the forward layers, the loss and
// the input-gradient products (dZ_l = dZ_{l+1} W_l * GELU'(Z_l)) without
// leaving the SM, organised as k_mlp_forward: operands in shared memory, two
// tiles per CTA in turn, weights streamed in both orientations.  What the
// weight gradients and the backward pass need goes to global memory: Z (FP32)
// as 16-byte blocks of four columns (a thread reads back what it wrote), A and
// dZ (BF16) with the batch as the contiguous k of the products, in k-blocks of
// 8 rows.  Bias gradients are summed per tile by a butterfly over the lanes.
//
// k_mlp_dw sums the five weight gradients dW_l = dZ_l^T A_{l-1} over slices of
// the batch, a CTA per (layer, slice), both 128-row halves of the product in
// TMEM, partial sums added to the gradient in FP32 four at a time.
//
// Layer by layer this was 16 launches of which most ran on 64 or 16 SMs and
// waited for scattered stores and 16-byte loads.  8,192 rows: 565 us of
// kernels, 73 + 20 us here (64 tiles: what bounds it is the latency of one
// tile's nine products and epilogues).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "cvx_mlp_tile.cuh"

namespace cvx {

namespace {

constexpr int kThreads = 640;
constexpr size_t kSmem = 2 * kABytes + kRing * kStageBytes + kW0Bytes + 2 * kW4Bytes +
                         kBiasFloats * sizeof(float) + 1024;

// Sums of 16 values per lane over the warp: lane 2 c (and 2 c + 1) returns the
// sum of column c' = bit-reversed place of the lane's upper four bits.
__device__ __forceinline__ float column_sum16(float (&v)[16], int lane, int &col) {
    col = 0;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const int o = 16 >> s, n = 8 >> s;  // exchange distance, values kept
        const bool up = (lane & o) != 0;
        col += up ? n : 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

}  // namespace

__global__ void __launch_bounds__(kThreads, 1) k_mlp_train(const MlpTrain f) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem =
        reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char *sA = smem;                  // two tiles' operands
    unsigned char *sB = sA + 2 * kABytes;      // ring of hidden-layer weights
    unsigned char *sW0 = sB + kRing * kStageBytes;
    unsigned char *sW4 = sW0 + kW0Bytes;       // last layer, forward
    unsigned char *sWt4 = sW4 + kW4Bytes;      // last layer, transposed
    float *sBias = reinterpret_cast<float *>(sWt4 + kW4Bytes);
    __shared__ __align__(8) uint64_t b_full[kRing], b_empty[kRing], w_full, a_ready[2], d_full[2], drain;
    __shared__ uint32_t s_tmem;
    __shared__ float s_db[4][kWidth], s_db4[8];  // bias gradients; the loss in s_db4[7]

    const int ntiles = (f.n + kRows - 1) / kRows;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int G = gridDim.x;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kRing; ++i) {
            mbar_init(&b_full[i], 1);
            mbar_init(&b_empty[i], 1);
        }
        mbar_init(&w_full, 1);
        mbar_init(&drain, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&a_ready[i], 16);
            mbar_init(&d_full[i], 1);
        }
        fence_mbar_init();
    }
    for (int i = threadIdx.x; i < kBiasFloats; i += kThreads)
        sBias[i] = i < 4 * kWidth ? f.bias[i >> 8][i & 255] : (i - 4 * kWidth < 7 ? f.bias[4][i - 4 * kWidth] : 0.0f);
    for (int i = threadIdx.x; i < 4 * kWidth; i += kThreads) s_db[i >> 8][i & 255] = 0.0f;
    if (threadIdx.x < 8) s_db4[threadIdx.x] = 0.0f;
    if (warp == 0) tmem_alloc(&s_tmem, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    // Products p of a tile: 0 input layer, 1-3 hidden layers, 4 outputs, 5 last
    // layer back, 6-8 hidden layers 3, 2, 1 back.  Tile g (0, 1) of a turn is
    // t0 + G g; the issuing warps and the epilogues walk the same sequence.
    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            int u = 0;  // ring stages issued
            mbar_expect_tx(&w_full, kW0Bytes + 2 * kW4Bytes);
            bulk_load(sW0, f.W[0], kW0Bytes, &w_full);
            bulk_load(sW4, f.W[4], kW4Bytes, &w_full);
            bulk_load(sWt4, f.Wt[4], kW4Bytes, &w_full);
            for (int t0 = blockIdx.x; t0 < ntiles && ok; t0 += 2 * G)
                for (int p = 1; p < 9 && ok; ++p) {
                    if (p == 4 || p == 5) continue;
                    const __nv_bfloat16 *w = p < 4 ? f.W[p] : f.Wt[9 - p];
                    for (int g = 0; g < 2 && ok; ++g) {
                        if (t0 + g * G >= ntiles) continue;
                        for (int c = 0; c < kWidth / kStageK; ++c, ++u) {
                            const int st = u % kRing, use = u / kRing;
                            if (use > 0 && !(ok = mbar_wait(&b_empty[st], (use - 1) & 1, kWaitNs))) break;
                            mbar_expect_tx(&b_full[st], kStageBytes);
                            bulk_load(sB + st * kStageBytes, w + (size_t)c * kStageK * kWidth,
                                      kStageBytes, &b_full[st]);
                        }
                    }
                }
            if (!ok) atomicExch(f.err, 1);
            mbar_wait(&w_full, 0, kWaitNs);
            drain_copies(b_full, kRing, u, kWaitNs);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t id_h = idesc_bf16(kRows, kWidth), id_o = idesc_bf16(kRows, kOutPad);
            bool ok = mbar_wait(&w_full, 0, kWaitNs);
            int u = 0, ph[2] = {0, 0};  // ring stages consumed, operands seen per tile
            for (int t0 = blockIdx.x; t0 < ntiles && ok; t0 += 2 * G)
                for (int p = 0; p < 9 && ok; ++p)
                    for (int g = 0; g < 2 && ok; ++g) {
                        if (t0 + g * G >= ntiles) continue;
                        if (!(ok = mbar_wait(&a_ready[g], ph[g] & 1, kWaitNs))) break;
                        ++ph[g];
                        tc_fence_after();
                        const uint32_t d = tmem + g * kWidth, a0 = smem_u32(sA + g * kABytes);
                        if (p == 0 || p == 5) {
                            umma_bf16(d, smem_desc(a0, kRows * 16, 128),
                                      smem_desc(smem_u32(p == 0 ? sW0 : sWt4), kWidth * 16, 128), id_h, 0u);
                        } else if (p == 4) {
                            for (int j = 0; j < kWidth / 16; ++j)
                                umma_bf16(d, smem_desc(a0 + 2 * j * kRows * 16, kRows * 16, 128),
                                          smem_desc(smem_u32(sW4) + 2 * j * kOutPad * 16, kOutPad * 16, 128),
                                          id_o, j > 0 ? 1u : 0u);
                        } else {
                            for (int c = 0; c < kWidth / kStageK; ++c, ++u) {
                                const int st = u % kRing, use = u / kRing;
                                if (!(ok = mbar_wait(&b_full[st], use & 1, kWaitNs))) break;
                                tc_fence_after();
                                const uint32_t b0 = smem_u32(sB + st * kStageBytes);
                                for (int j = 0; j < kStageK / 16; ++j) {
                                    const int kb = c * (kStageK / 8) + 2 * j;
                                    umma_bf16(d, smem_desc(a0 + kb * kRows * 16, kRows * 16, 128),
                                              smem_desc(b0 + 2 * j * kWidth * 16, kWidth * 16, 128), id_h,
                                              c > 0 || j > 0 ? 1u : 0u);
                                }
                                umma_commit(&b_empty[st]);
                            }
                            if (!ok) break;
                        }
                        umma_commit(&d_full[g]);
                    }
            if (!ok) atomicExch(f.err, 1);
            drain_mmas(&drain, kWaitNs);
        }
    } else if (warp >= 4) {
        // columns 64 part .. 64 part + 63 of the rows of TMEM lanes 32 quarter ..
        const int quarter = warp & 3, part = (warp - 4) >> 2;
        const int row = 32 * quarter + lane;
        unsigned char *A0 = sA + row * 16;  // k-block kb at + kb * kRows * 16
        const uint32_t trow = tmem + ((uint32_t)(32 * quarter) << 16);
        const float inv_n = 1.0f / (float)f.n;
        bool ok = true;
        int ph[2] = {0, 0};  // accumulators read per tile
        auto ready = [&](int g) {
            fence_proxy_async();  // the operand is read by the async proxy
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&a_ready[g]);
        };
        // 8 values of row m to columns c .. c + 7 of a batch-major matrix of w
        // columns: element (m, c) at ((m / 8) w + c) 8 + m % 8
        auto store_t = [&](__nv_bfloat16 *T, int w, long long m, int c, uint4 x) {
            __nv_bfloat16 *d = T + ((m >> 3) * w + c) * 8 + (m & 7);
            const uint32_t v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int k = 0; k < 8; ++k)
                d[8 * k] = __ushort_as_bfloat16((unsigned short)(v[k >> 1] >> (16 * (k & 1))));
        };
        for (int t0 = blockIdx.x; t0 < ntiles && ok; t0 += 2 * G) {
            const int ng = t0 + G < ntiles ? 2 : 1;
            // ---- the input operands: standardised features, zero-padded to 16
            for (int g = 0; g < ng; ++g) {
                const long long m = (long long)(t0 + g * G) * kRows + row;
                if (part < 2) {
                    uint4 x = make_uint4(0u, 0u, 0u, 0u);
                    if (m < f.n && part == 0) {
                        const float *r = f.X + 6 * (f.idx ? (long long)f.idx[m] : m);
                        uint32_t w[3];
#pragma unroll
                        for (int k = 0; k < 3; ++k)
                            w[k] = pack_bf16(pk2((r[2 * k] - f.scale[2 * k]) * f.scale[6 + 2 * k],
                                                 (r[2 * k + 1] - f.scale[2 * k + 1]) * f.scale[7 + 2 * k]));
                        x = make_uint4(w[0], w[1], w[2], 0u);
                    }
                    *reinterpret_cast<uint4 *>(A0 + g * kABytes + part * kRows * 16) = x;
                    store_t(f.XT, kInPad, m, 8 * part, x);
                }
                ready(g);
            }
            for (int p = 0; p < 9 && ok; ++p)
                for (int g = 0; g < ng; ++g) {
                    if (!(ok = mbar_wait_warp(&d_full[g], ph[g] & 1, kWaitNs))) break;
                    ++ph[g];
                    tc_fence_after();
                    const long long m = (long long)(t0 + g * G) * kRows + row;
                    const bool in = m < f.n;
                    unsigned char *A = A0 + g * kABytes + 8 * part * kRows * 16;
                    if (p < 4) {
                        // ---- hidden layer p: z, GELU, the next operand
                        const float *bias = sBias + p * kWidth + 64 * part;
                        float4 *Z = reinterpret_cast<float4 *>(f.Z[p]) + (size_t)16 * part * f.ld + m;
#pragma unroll
                        for (int c = 0; c < 64; c += 32) {
                            uint32_t v[32];
                            tmem_ld32(trow + g * kWidth + 64 * part + c, v);
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                uint32_t w[4];
                                float z[8];
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    const float2 b = *reinterpret_cast<const float2 *>(bias + c + 8 * k + 2 * i);
                                    const f32x2 zz = add2(pk2(__uint_as_float(v[8 * k + 2 * i]),
                                                              __uint_as_float(v[8 * k + 2 * i + 1])),
                                                          pk2(b.x, b.y));
                                    upk2(zz, z[2 * i], z[2 * i + 1]);
                                    w[i] = gelu2_bf16(zz);
                                }
                                Z[(size_t)(c / 4 + 2 * k) * f.ld] = make_float4(z[0], z[1], z[2], z[3]);
                                Z[(size_t)(c / 4 + 2 * k + 1) * f.ld] = make_float4(z[4], z[5], z[6], z[7]);
                                const uint4 x = make_uint4(w[0], w[1], w[2], w[3]);
                                *reinterpret_cast<uint4 *>(A + (c / 8 + k) * kRows * 16) = x;
                                store_t(f.AT[p], kWidth, m, 64 * part + c + 8 * k, x);
                            }
                        }
                        ready(g);
                    } else if (p == 4) {
                        // ---- outputs, loss, dL/d(out): the next operand (16 wide)
                        uint4 x = make_uint4(0u, 0u, 0u, 0u);
                        if (part == 0) {
                            float v[16], gr[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                            tmem_ld16(trow + g * kWidth, v);
                            float L = 0.0f;
                            if (in) {
                                const float *y = f.Y + 7 * (f.idx ? (long long)f.idx[m] : m);
                                float o[7];
#pragma unroll
                                for (int k = 0; k < 7; ++k) o[k] = v[k] + sBias[4 * kWidth + k];
                                if (!isnan(y[0])) {
                                    for (int i = 0; i < 2; ++i) {
                                        const float d = 2.0f * (o[i] - y[i]);
                                        L += 1.0f - cosf(d);
                                        gr[i] = 2.0f * sinf(d);
                                    }
                                }
                                if (!isnan(y[2])) {
                                    const float s = 1.0f / (1.0f + expf(-o[2]));
                                    L += (s - y[2]) * (s - y[2]);
                                    gr[2] = 2.0f * (s - y[2]) * s * (1.0f - s);
                                }
                                for (int j = 3; j < 7; ++j) {
                                    const float d = o[j] - y[j];
                                    L += d * d;
                                    gr[j] = 2.0f * d;
                                }
                            }
                            x = make_uint4(pack_bf16(pk2(gr[0] * inv_n, gr[1] * inv_n)),
                                           pack_bf16(pk2(gr[2] * inv_n, gr[3] * inv_n)),
                                           pack_bf16(pk2(gr[4] * inv_n, gr[5] * inv_n)),
                                           pack_bf16(pk2(gr[6] * inv_n, 0.0f)));
                            gr[7] = L;
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                for (int o = 16; o; o >>= 1) gr[k] += __shfl_xor_sync(0xffffffffu, gr[k], o);
                                if (lane == 0) atomicAdd(&s_db4[k], gr[k]);
                            }
                        }
                        if (part < 2) {
                            *reinterpret_cast<uint4 *>(A0 + g * kABytes + part * kRows * 16) = x;
                            store_t(f.dZoT, kOutPad, m, 8 * part, x);
                        }
                        ready(g);
                    } else {
                        // ---- dZ of hidden layer l = 8 - p, the next operand
                        const int l = 8 - p;
                        const float4 *Z = reinterpret_cast<const float4 *>(f.Z[l]) + (size_t)16 * part * f.ld + m;
#pragma unroll 1
                        for (int c = 0; c < 64; c += 32) {
                            uint32_t v[32];
                            tmem_ld32(trow + g * kWidth + 64 * part + c, v);
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                float dz[16];
#pragma unroll
                                for (int k = 0; k < 4; ++k) {
                                    const float4 z = Z[(size_t)(c / 4 + 4 * h + k) * f.ld];
                                    const f32x2 d0 = mul2(pk2(__uint_as_float(v[16 * h + 4 * k]),
                                                              __uint_as_float(v[16 * h + 4 * k + 1])),
                                                          gelu_grad2(pk2(z.x, z.y)));
                                    const f32x2 d1 = mul2(pk2(__uint_as_float(v[16 * h + 4 * k + 2]),
                                                              __uint_as_float(v[16 * h + 4 * k + 3])),
                                                          gelu_grad2(pk2(z.z, z.w)));
                                    upk2(d0, dz[4 * k], dz[4 * k + 1]);
                                    upk2(d1, dz[4 * k + 2], dz[4 * k + 3]);
                                }
                                if (!in)
                                    for (int k = 0; k < 16; ++k) dz[k] = 0.0f;
#pragma unroll
                                for (int k = 0; k < 2; ++k) {
                                    const uint4 x = make_uint4(pack_bf16(pk2(dz[8 * k], dz[8 * k + 1])),
                                                               pack_bf16(pk2(dz[8 * k + 2], dz[8 * k + 3])),
                                                               pack_bf16(pk2(dz[8 * k + 4], dz[8 * k + 5])),
                                                               pack_bf16(pk2(dz[8 * k + 6], dz[8 * k + 7])));
                                    *reinterpret_cast<uint4 *>(A + (c / 8 + 2 * h + k) * kRows * 16) = x;
                                    store_t(f.dZT[l], kWidth, m, 64 * part + c + 16 * h + 8 * k, x);
                                }
                                int col;
                                const float sum = column_sum16(dz, lane, col);
                                if (!(lane & 1)) atomicAdd(&s_db[l][64 * part + c + 16 * h + col], sum);
                            }
                        }
                        if (p < 8) {
                            ready(g);
                        } else {
                            tc_fence_before();
                            __syncwarp();
                        }
                    }
                }
        }
        if (!ok && lane == 0) atomicExch(f.err, 1);
    }
    tc_fence_before();
    __syncthreads();
    for (int i = threadIdx.x; i < 4 * kWidth; i += kThreads)
        atomicAdd(f.dbias[i >> 8] + (i & 255), s_db[i >> 8][i & 255]);
    if (threadIdx.x < 7) atomicAdd(f.dbias[4] + threadIdx.x, s_db4[threadIdx.x] * (1.0f / (float)f.n));
    if (threadIdx.x == 7) atomicAdd(f.loss, s_db4[7] * (1.0f / (float)f.n));
    if (warp == 0) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

namespace {

constexpr int kDwRing = 3, kDwK = 64;                            // stages, batch rows per stage
constexpr int kDwABytes = kWidth * kDwK * 2, kDwStage = 2 * kDwABytes;  // 32 KB each operand
constexpr size_t kDwSmem = (size_t)kDwRing * kDwStage + 1024;
constexpr int kDwThreads = 384;

}  // namespace

// One CTA per (slice of the batch, layer): D = dZ^T A over its rows.  Jobs 0-2:
// hidden layers 1-3, D[out][in]; job 3: the last layer as D[in][out 16]; job 4:
// the input layer, D[out][in 16].  Warp 0 loads, warp 1 multiplies, warps 4-11
// add the result.
__global__ void __launch_bounds__(kDwThreads, 1) k_mlp_dw(const MlpTrain f, int chunks) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem =
        reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full[kDwRing], empty[kDwRing], done, drain;
    __shared__ uint32_t s_tmem;
    const int job = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c0 = (int)((long long)chunks * blockIdx.x / gridDim.x);
    const int c1 = (int)((long long)chunks * (blockIdx.x + 1) / gridDim.x);
    if (c0 >= c1) return;
    const int NB = job < 3 ? kWidth : 16;  // rows of the second operand
    const __nv_bfloat16 *A = job < 3 ? f.dZT[job + 1] : (job == 3 ? f.AT[3] : f.dZT[0]);
    const __nv_bfloat16 *B = job < 3 ? f.AT[job] : (job == 3 ? f.dZoT : f.XT);
    const unsigned bbytes = (unsigned)NB * kDwK * 2;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kDwRing; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        mbar_init(&done, 1);
        mbar_init(&drain, 1);
        fence_mbar_init();
    }
    if (warp == 0) tmem_alloc(&s_tmem, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            int u = 0;
            for (int c = c0; c < c1; ++c, ++u) {
                const int st = u % kDwRing, use = u / kDwRing;
                if (use > 0 && !(ok = mbar_wait(&empty[st], (use - 1) & 1, kWaitNs))) break;
                unsigned char *d = smem + st * kDwStage;
                mbar_expect_tx(&full[st], kDwABytes + bbytes);
                bulk_load(d, A + (size_t)c * kDwK * kWidth, kDwABytes, &full[st]);
                bulk_load(d + kDwABytes, B + (size_t)c * kDwK * NB, bbytes, &full[st]);
            }
            if (!ok) atomicExch(f.err, 1);
            drain_copies(full, kDwRing, u, kWaitNs);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t id = idesc_bf16(kRows, NB);
            bool ok = true;
            int u = 0;
            for (int c = c0; c < c1; ++c, ++u) {
                const int st = u % kDwRing, use = u / kDwRing;
                if (!(ok = mbar_wait(&full[st], use & 1, kWaitNs))) break;
                tc_fence_after();
                const uint32_t a0 = smem_u32(smem + st * kDwStage), b0 = a0 + kDwABytes;
                for (int j = 0; j < kDwK / 16; ++j)
                    for (int h = 0; h < 2; ++h)
                        umma_bf16(tmem + h * kWidth,
                                  smem_desc(a0 + 2 * j * kWidth * 16 + h * kRows * 16, kWidth * 16, 128),
                                  smem_desc(b0 + 2 * j * NB * 16, NB * 16, 128), id,
                                  u > 0 || j > 0 ? 1u : 0u);
                umma_commit(&empty[st]);
            }
            if (ok) umma_commit(&done);
            else atomicExch(f.err, 1);
            drain_mmas(&drain, kWaitNs);
        }
    } else if (warp >= 4) {
        const int quarter = warp & 3, h = (warp - 4) >> 2;
        const int r = kRows * h + 32 * quarter + lane;
        const uint32_t trow = tmem + h * kWidth + ((uint32_t)(32 * quarter) << 16);
        if (mbar_wait_warp(&done, 0, kWaitNs)) {
            tc_fence_after();
            if (job < 3) {
                float4 *g = reinterpret_cast<float4 *>(f.dW[job + 1] + (size_t)r * kWidth);
                for (int c = 0; c < kWidth; c += 32) {
                    uint32_t v[32];
                    tmem_ld32(trow + c, v);
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        atomicAdd(g + c / 4 + k,
                                  make_float4(__uint_as_float(v[4 * k]), __uint_as_float(v[4 * k + 1]),
                                              __uint_as_float(v[4 * k + 2]), __uint_as_float(v[4 * k + 3])));
                }
            } else {
                float v[16];
                tmem_ld16(trow, v);
                if (job == 3) {
#pragma unroll
                    for (int k = 0; k < 7; ++k) atomicAdd(f.dW[4] + k * kWidth + r, v[k]);
                } else {
#pragma unroll
                    for (int k = 0; k < 6; ++k) atomicAdd(f.dW[0] + 6 * r + k, v[k]);
                }
            }
        } else if (lane == 0) {
            atomicExch(f.err, 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

cudaError_t launch_mlp_grad(const MlpTrain &f, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_mlp_dw, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDwSmem);
    if (e != cudaSuccess) return e;
    const int tiles = (f.n + kRows - 1) / kRows;
    k_mlp_train<<<(unsigned)std::min(tiles, sms), kThreads, kSmem, s>>>(f);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // slices: eight stages or more each (a slice ends in 65,536 additions per
    // layer), one wave of CTAs at most
    const int chunks = 2 * tiles;
    const int slices = std::max(1, std::min(chunks / 8, sms / 5));
    k_mlp_dw<<<dim3((unsigned)slices, 5), kDwThreads, kDwSmem, s>>>(f, chunks);
    return cudaGetLastError();
}

}  // namespace cvx
