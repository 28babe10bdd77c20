// cvx_refine.cuh -- integer keys of FP64 values, shared by the refinement
// kernels.
//
// The minima of v - s x are compared as order-preserving integer keys of the
// doubles, so that the comparisons run on the integer pipe: the FP64 pipe
// (2 lanes per SM per clock) is what bounds the refinement, and a key compares
// exactly as its double does.
#pragma once

#include "cvx_bridge.cuh"

namespace cvx {

// Integer key of a double that is not NaN: x < y iff dkey(x) < dkey(y), and
// x == y iff the keys are equal (-0 and +0 share the key 0).
__device__ __forceinline__ long long dkey(double x) {
    const long long b = __double_as_longlong(x);
    return b >= 0 ? b : -(b & 0x7fffffffffffffffLL);
}

constexpr long long kKeyInf = 0x7ff0000000000000LL;  // dkey(+inf)

// Warp-wide minimum of (key, sample index); ties to the lower index if
// prefer_low, else to the higher.
__device__ __forceinline__ void warp_min_key(long long &v, int &k, bool prefer_low) {
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const long long v2 = __shfl_xor_sync(kFull, v, o);
        const int k2 = __shfl_xor_sync(kFull, k, o);
        if (v2 < v || (v2 == v && (prefer_low ? k2 < k : k2 > k))) {
            v = v2;
            k = k2;
        }
    }
}

}  // namespace cvx
