// cvx_mlp_fused.cu -- inference of the surrogate network in one kernel: all
// five layers of a tile of 128 rows without leaving the SM.
//
// The layer-by-layer form (cvx_gemm.cu) writes and reads 128 KB of activations
// per tile and layer and spent 46 us per layer of 65,536 rows, three times
// what its epilogue needs.  Here a CTA works on two tiles at a time.  Per tile
// the activations stay in one 64 KB shared-memory operand (the epilogue of a
// layer writes the next layer's A operand in place, k-blocks of 8 elements x
// 128 rows x 16 bytes as in cvx_tc.cuh) and the accumulator in 256 TMEM
// columns; the weights of the three hidden layers (128 KB each, from L2)
// stream through a ring of four 16 KB stages by bulk copies of a copy packed in
// that layout, once per tile and layer.
// The MMAs of one tile run while the other tile's epilogue does.
//
// What bounds it: instruction issue in the epilogue (10.5 instructions per
// activation, its arithmetic paired: fma.rn.f32x2) and the turns between MMAs
// and epilogues.  1,000,000 rows: 3.54 ms layer by layer, 0.68 ms here.  The
// weights by tensor-map boxes of 16-byte rows took 0.94 ms (the box engine
// takes a row at a time), one pass of the weights for both tiles 0.91 ms (the
// epilogues wait for both tiles' MMAs), eight epilogue warps per tile instead
// of all sixteen on each in turn 0.74 ms.
//
// Warp 0 (lane 0) issues the bulk copies, warp 1 (lane 0) the MMAs, warps 4-19
// are the epilogue of either tile in turn (four threads per row, 64 columns
// each).  Every wait is bounded.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "cvx_mlp_tile.cuh"

namespace cvx {

namespace {

constexpr size_t kSmem = 2 * kABytes + kRing * kStageBytes + kW0Bytes + kW4Bytes +
                         kBiasFloats * sizeof(float) + 1024;
constexpr int kThreads = 640;

}  // namespace

__global__ void __launch_bounds__(kThreads, 1)
    k_mlp_forward(const MlpForward f) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem =
        reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char *sA = smem;                            // two tiles' A operands
    unsigned char *sB = sA + 2 * kABytes;                // ring of hidden-layer weights
    unsigned char *sW0 = sB + kRing * kStageBytes;
    unsigned char *sW4 = sW0 + kW0Bytes;
    float *sBias = reinterpret_cast<float *>(sW4 + kW4Bytes);
    __shared__ __align__(8) uint64_t b_full[kRing], b_empty[kRing], w_full, a_ready[2], d_full[2], drain;
    __shared__ uint32_t s_tmem;

    const int Mv = f.M_dev ? min(*f.M_dev - f.m_off, f.M) : f.M;
    const int ntiles = Mv > 0 ? (Mv + kRows - 1) / kRows : 0;
    if ((int)blockIdx.x >= ntiles) return;
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
    if (warp == 0) tmem_alloc(&s_tmem, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    // Tile g (0, 1) of turn `it` of this CTA is blockIdx.x + G (2 it + g); both
    // issuing warps and the epilogues walk the same sequence of tiles.
    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            int u = 0;  // ring stages issued
            mbar_expect_tx(&w_full, kW0Bytes + kW4Bytes);
            bulk_load(sW0, f.W[0], kW0Bytes, &w_full);
            bulk_load(sW4, f.W[4], kW4Bytes, &w_full);
            for (int t0 = blockIdx.x; t0 < ntiles && ok; t0 += 2 * G)
                for (int l = 1; l < 4 && ok; ++l)
                    for (int g = 0; g < 2 && ok; ++g) {
                        if (t0 + g * G >= ntiles) continue;
                        for (int c = 0; c < kWidth / kStageK; ++c, ++u) {
                            const int st = u % kRing, use = u / kRing;
                            if (use > 0 && !(ok = mbar_wait(&b_empty[st], (use - 1) & 1, kWaitNs))) break;
                            mbar_expect_tx(&b_full[st], kStageBytes);
                            bulk_load(sB + st * kStageBytes,
                                      f.W[l] + (size_t)c * kStageK * kWidth, kStageBytes, &b_full[st]);
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
                for (int l = 0; l < 5 && ok; ++l)
                    for (int g = 0; g < 2 && ok; ++g) {
                        if (t0 + g * G >= ntiles) continue;
                        if (!(ok = mbar_wait(&a_ready[g], ph[g] & 1, kWaitNs))) break;
                        ++ph[g];
                        tc_fence_after();
                        const uint32_t d = tmem + g * kWidth, a0 = smem_u32(sA + g * kABytes);
                        if (l == 0) {
                            umma_bf16(d, smem_desc(a0, kRows * 16, 128),
                                      smem_desc(smem_u32(sW0), kWidth * 16, 128), id_h, 0u);
                        } else if (l == 4) {
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
        bool ok = true;
        int ph[2] = {0, 0};  // accumulators read per tile
        auto ready = [&](int g) {
            fence_proxy_async();  // the operand is read by the async proxy
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&a_ready[g]);
        };
        for (int t0 = blockIdx.x; t0 < ntiles && ok; t0 += 2 * G) {
            const int ng = t0 + G < ntiles ? 2 : 1;
            // ---- the input operands: standardised features, zero-padded to 16
            for (int g = 0; g < ng; ++g) {
                const long long m = (long long)(t0 + g * G) * kRows + row;
                if (part < 2) {
                    uint4 x = make_uint4(0u, 0u, 0u, 0u);
                    if (m < Mv) {
                        if (f.X16) {
                            x = *reinterpret_cast<const uint4 *>(f.X16 + m * kInPad + 8 * part);
                        } else if (part == 0) {
                            const float *r = f.X + 6 * m;
                            uint32_t w[3];
#pragma unroll
                            for (int k = 0; k < 3; ++k) {
                                const __nv_bfloat162 h = __floats2bfloat162_rn(
                                    (r[2 * k] - f.scale[2 * k]) * f.scale[6 + 2 * k],
                                    (r[2 * k + 1] - f.scale[2 * k + 1]) * f.scale[7 + 2 * k]);
                                w[k] = *reinterpret_cast<const uint32_t *>(&h);
                            }
                            x = make_uint4(w[0], w[1], w[2], 0u);
                        }
                    }
                    *reinterpret_cast<uint4 *>(A0 + g * kABytes + part * kRows * 16) = x;
                }
                ready(g);
            }
            // ---- hidden layers: bias, GELU, the next operand
            for (int l = 0; l < 4 && ok; ++l)
                for (int g = 0; g < ng; ++g) {
                    if (!(ok = mbar_wait_warp(&d_full[g], ph[g] & 1, kWaitNs))) break;
                    ++ph[g];
                    tc_fence_after();
                    const float *bias = sBias + l * kWidth + 64 * part;
                    unsigned char *A = A0 + g * kABytes + 8 * part * kRows * 16;
#pragma unroll
                    for (int c = 0; c < 64; c += 32) {
                        uint32_t v[32];
                        tmem_ld32(trow + g * kWidth + 64 * part + c, v);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            uint32_t w[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const float2 b = *reinterpret_cast<const float2 *>(bias + c + 8 * k + 2 * i);
                                w[i] = gelu2_bf16(add2(pk2(__uint_as_float(v[8 * k + 2 * i]),
                                                           __uint_as_float(v[8 * k + 2 * i + 1])),
                                                       pk2(b.x, b.y)));
                            }
                            *reinterpret_cast<uint4 *>(A + (c / 8 + k) * kRows * 16) =
                                make_uint4(w[0], w[1], w[2], w[3]);
                        }
                    }
                    ready(g);
                }
            // ---- outputs
            for (int g = 0; g < ng && ok; ++g) {
                if (!(ok = mbar_wait_warp(&d_full[g], ph[g] & 1, kWaitNs))) break;
                ++ph[g];
                tc_fence_after();
                if (part == 0) {
                    float v[16];
                    tmem_ld16(trow + g * kWidth, v);
                    const long long m = (long long)(t0 + g * G) * kRows + row;
                    if (m < Mv) {
                        float *o = f.out + 7 * m;
#pragma unroll
                        for (int k = 0; k < 7; ++k) o[k] = v[k] + sBias[4 * kWidth + k];
                    }
                }
                tc_fence_before();
                __syncwarp();
            }
        }
        if (!ok && lane == 0) atomicExch(f.err, 1);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

cudaError_t launch_mlp_forward(const MlpForward &f, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kSmem);
    if (e != cudaSuccess) return e;
    const int tiles = (f.M + kRows - 1) / kRows;
    k_mlp_forward<<<(unsigned)std::max(1, std::min(tiles, sms)), kThreads, kSmem, s>>>(f);
    return cudaGetLastError();
}

}  // namespace cvx
