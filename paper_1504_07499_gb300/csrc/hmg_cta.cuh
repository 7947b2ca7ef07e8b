// CTA shapes and sums shared by the FP64 and FP32 pass kernels that take their sizes at compile time.
#pragma once

#include <cuda_runtime.h>

namespace hmg {

// largest divisor of n that is at most lim
constexpr int divisor_upto(long long n, int lim) {
    int d = 1;
    for (int i = 1; i <= lim; ++i)
        if (n % i == 0) d = i;
    return d;
}
constexpr int pow2_at_least(int n) {
    int p = 1;
    while (p < n) p *= 2;
    return p;
}
// fixed-order sum over the CTA's T threads, valid in thread 0; sh: pow2_at_least(T) doubles
template <int T>
__device__ double cta_sum(double v, double* sh) {
    constexpr int P = pow2_at_least(T);
    sh[threadIdx.x] = v;
    if (threadIdx.x + T < P) sh[threadIdx.x + T] = 0.0;
    __syncthreads();
    for (int s = P / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    return sh[0];
}

}  // namespace hmg
