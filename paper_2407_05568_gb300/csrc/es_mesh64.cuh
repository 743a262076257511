// es_mesh64.cuh -- maxima of non-negative doubles by their ordered bits (comparisons of doubles and
// fmax/fmin take the FP64 pipe), for the FP64 mesh and time-step kernels, and the limiter's test.
#pragma once
#include <cuda_runtime.h>

namespace es {

// 2 (1 + 2^-50): the limiter forms room/(2 |dx|) where room < m (LIMIT_TEST |dx|)
constexpr double LIMIT_TEST = 2.0 + 0x1p-49;

// max(a, b), a >= 0, b >= 0 or NaN (a NaN is passed over, as fmax does)
__device__ __forceinline__ double max_bits(double a, double b) {
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    return y > x && y <= 0x7ff0000000000000LL ? b : a;
}

// the block's maxima of N such values, on thread 0
template <int N>
__device__ __forceinline__ void block_max_bits(double* v) {
    __shared__ double sh[N][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        for (int o = 16; o > 0; o >>= 1) v[k] = max_bits(v[k], __shfl_xor_sync(0xffffffffu, v[k], o));
        if (lane == 0) sh[k][w] = v[k];
    }
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            v[k] = lane < nw ? sh[k][lane] : 0.0;
            for (int o = 16; o > 0; o >>= 1) v[k] = max_bits(v[k], __shfl_xor_sync(0xffffffffu, v[k], o));
        }
    }
}

}  // namespace es
