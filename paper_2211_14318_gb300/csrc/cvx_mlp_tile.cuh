// cvx_mlp_tile.cuh -- what the network's tile kernels (inference, training)
// share: a tile of 128 rows whose operands lie in shared memory as k-blocks of
// 8 elements x rows x 16 bytes (cvx_tc.cuh), weights packed in that layout, and
// the paired arithmetic of the GELU.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "cvx_device.cuh"
#include "cvx_mlp.h"
#include "cvx_tc.cuh"

namespace cvx {

constexpr int kRows = 128, kWidth = 256, kOutPad = 16, kInPad = 16;
constexpr int kRing = 4, kStageK = 32;                       // stages, k per stage
constexpr int kStageBytes = kWidth * kStageK * 2;            // 16 KB
constexpr int kABytes = kRows * kWidth * 2;                  // 64 KB
constexpr int kW0Bytes = kWidth * kInPad * 2, kW4Bytes = kOutPad * kWidth * 2;
constexpr int kBiasFloats = 4 * kWidth + kOutPad;
constexpr uint64_t kWaitNs = 1000000000ull;  // 1 s per wait, then give up

__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Normal CDF Phi(z) of two values and e^{-z^2 / 2}, erf from Abramowitz &
// Stegun, Handbook of Mathematical Functions, formula 7.1.26:
//   erf(x) = 1 - (a1 t + a2 t^2 + a3 t^3 + a4 t^4 + a5 t^5) exp(-x^2),
//   t = 1 / (1 + p x), x >= 0, |error| <= 1.5e-7.
__device__ __forceinline__ f32x2 normal_cdf2(f32x2 z, f32x2 &ex) {
    auto c2 = [](float c) { return pk2(c, c); };
    float z0, z1, x0, x1;
    upk2(z, z0, z1);
    const f32x2 x = mul2(pk2(fabsf(z0), fabsf(z1)), c2(0.70710678118654752f));
    float d0, d1;
    upk2(fma2(c2(0.3275911f), x, c2(1.0f)), d0, d1);
    const f32x2 t = pk2(rcp_approx(d0), rcp_approx(d1));
    // minus the polynomial: all coefficients negated
    f32x2 p = fma2(t, c2(-1.061405429f), c2(1.453152027f));
    p = fma2(t, p, c2(-1.421413741f));
    p = fma2(t, p, c2(0.284496736f));
    p = mul2(t, fma2(t, p, c2(-0.254829592f)));
    upk2(mul2(mul2(x, x), c2(-1.4426950408889634f)), x0, x1);
    ex = pk2(ex2_approx(x0), ex2_approx(x1));
    float e0, e1;
    upk2(fma2(p, ex, c2(1.0f)), e0, e1);  // erf(x)
    return fma2(c2(0.5f), pk2(copysignf(e0, z0), copysignf(e1, z1)), c2(0.5f));
}

__device__ __forceinline__ uint32_t pack_bf16(f32x2 a) {
    float a0, a1;
    upk2(a, a0, a1);
    const __nv_bfloat162 h = __floats2bfloat162_rn(a0, a1);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// GELU z Phi(z) of two activations, packed to BF16.
__device__ __forceinline__ uint32_t gelu2_bf16(f32x2 z) {
    f32x2 ex;
    return pack_bf16(mul2(z, normal_cdf2(z, ex)));
}

// GELU'(z) = Phi(z) + z phi(z), phi the normal density.
__device__ __forceinline__ f32x2 gelu_grad2(f32x2 z) {
    f32x2 ex;
    const f32x2 P = normal_cdf2(z, ex);
    const f32x2 phi = mul2(pk2(0.39894228040143268f, 0.39894228040143268f), ex);
    return fma2(z, phi, P);
}

// Contiguous bytes, global to shared memory (both 16-byte aligned, a multiple
// of 16 bytes).
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// 32 consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

}  // namespace cvx
