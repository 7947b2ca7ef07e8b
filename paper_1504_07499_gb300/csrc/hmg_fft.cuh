// Complex helpers and the radix-2, 3, 4 and 8 butterflies of the FP32 register transforms.
// The inverse transforms use the conjugate twiddles and butterflies (no scaling).
#pragma once

#include <cuda_runtime.h>
#include "hmg_internal.h"

namespace hmg {

__device__ __forceinline__ float2 mk(float a, float b) { return make_float2(a, b); }

template <typename T2> __device__ __forceinline__ T2 cmul(T2 a, T2 b) {
    return mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * conj(b)
template <typename T2> __device__ __forceinline__ T2 cmulc(T2 a, T2 b) {
    return mk(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
template <typename T2> __device__ __forceinline__ T2 cconj(T2 a) { return mk(a.x, -a.y); }
// multiply by -i (forward) or +i (inverse)
template <bool FWD, typename T2> __device__ __forceinline__ T2 mul_mi(T2 a) {
    return FWD ? mk(a.y, -a.x) : mk(-a.y, a.x);
}

// FP32 complex adds and subtracts as single packed two-lane FP32 instructions (sm_100
// and later); a - b is b * (-1) + a, exact product, one rounding, as the scalar form.
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// Radix-R DFT in registers, forward sign exp(-2 pi i/R) or its conjugate.
template <bool FWD, typename T2> __device__ __forceinline__ void bfly2(T2* v) {
    T2 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
}

template <bool FWD, typename T2> __device__ __forceinline__ void bfly4(T2* v) {
    T2 t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
    T2 t2 = cadd(v[1], v[3]), t3 = mul_mi<FWD>(csub(v[1], v[3]));
    v[0] = cadd(t0, t2);
    v[2] = csub(t0, t2);
    v[1] = cadd(t1, t3);
    v[3] = csub(t1, t3);
}

template <bool FWD, typename T2> __device__ __forceinline__ void bfly3(T2* v) {
    using S = decltype(v[0].x);
    const S h = S(0.86602540378443864676);  // sin(2 pi / 3)
    T2 t = cadd(v[1], v[2]);
    T2 u = csub(v[1], v[2]);
    T2 m = mk(v[0].x - S(0.5) * t.x, v[0].y - S(0.5) * t.y);
    // forward: X1 = m - i h u, X2 = m + i h u
    T2 iu = mul_mi<FWD>(u);  // -i u (forward) / +i u (inverse)
    v[0] = cadd(v[0], t);
    v[1] = mk(m.x + h * iu.x, m.y + h * iu.y);
    v[2] = mk(m.x - h * iu.x, m.y - h * iu.y);
}

template <bool FWD, typename T2> __device__ __forceinline__ void bfly8(T2* v) {
    using S = decltype(v[0].x);
    const S c = S(0.70710678118654752440);  // cos(pi/4)
    T2 a[4], b[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        a[r] = cadd(v[r], v[r + 4]);
        b[r] = csub(v[r], v[r + 4]);
    }
    // b_r *= w8^r, w8 = exp(-i pi/4) forward
    b[1] = FWD ? mk(c * (b[1].x + b[1].y), c * (b[1].y - b[1].x))
               : mk(c * (b[1].x - b[1].y), c * (b[1].y + b[1].x));
    b[2] = mul_mi<FWD>(b[2]);
    b[3] = FWD ? mk(c * (b[3].y - b[3].x), -c * (b[3].x + b[3].y))
               : mk(-c * (b[3].x + b[3].y), c * (b[3].x - b[3].y));
    bfly4<FWD>(a);
    bfly4<FWD>(b);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        v[2 * r] = a[r];
        v[2 * r + 1] = b[r];
    }
}

}  // namespace hmg
