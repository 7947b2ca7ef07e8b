// FFT passes of one Eyre-Milton sweep (§3 Algorithm, steps 2-7) and the helpers
// around them.  The 3D real transform runs as five passes over HBM:
//   x forward (real->complex, polarization of step 2 fused on load),
//   y forward,
//   z forward + Green operator of step 4 (+ macroscopic gradient at DC) + z inverse,
//   y inverse,
//   x inverse (complex->real) with the update of step 7 written out and the
//   step-6 residual accumulated in FP64.
// The sweep is written in the polarization variable tau = (k + k0) e: with
// Y = (k - k0)/(k + k0) and P the projector xi xi^T/|xi|^2 (Gamma0 = -P/k0 for
// L0 = -k0 I), steps 2-7 read tau^{n+1} = (I - 2P)(Y tau^n) + 2 k0 E, and
// e^n - e_comp^n = (tau^n - tau^{n+1}) / (2 k0), so no field but tau is stored.
// (The basic scheme runs through the same passes on e itself, with its own Y and the
// Green step -P; GridDesc carries the scheme's coefficients.)  The pass kernels are in
// hmg_fast.cu and hmg_gen32_kernels.cuh (FP32) and hmg_fixed_kernels.cuh (FP64); this file
// holds their dispatch by precision and size, the reductions and the pointwise helpers.
//
// Spectrum layout: after the x pass each row of N reals becomes N/2 complex values
// (x-major rows, same byte size as the real field); entry kx = 0 packs the two real
// planes kx = 0 and kx = N/2 as X(0) + i X(N/2).  The y and z passes transform that
// packed column like any other; the Green operator treats its four special modes
// (ky, kz in {0, N/2}) by real and imaginary part.
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <type_traits>

#include "hmg_internal.h"
#include "hmg_launch.cuh"

namespace hmg {

// ---------------------------------------------------------------------------
// small device helpers
// ---------------------------------------------------------------------------

// Fixed-order CTA sum of one double per thread (T threads); result valid in thread 0.
template <int T>
__device__ double block_sum(double v, double* sh) {
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int s = T / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    return sh[0];
}

// ---------------------------------------------------------------------------
// reductions and pointwise helpers
// ---------------------------------------------------------------------------

// Sum of the CTA partials of one slot (and group) by one CTA.  The chain of dependent FP64 adds
// per thread is what it waits for, so large counts take 1024 threads (12 288 partials at 256^3:
// 42 us with 256 threads) and small ones 256 (the tree over 1024 threads alone takes longer).
// With stop.flags, a sweep residual also decides whether its slot goes on: the slot's flag is
// cleared once the sum is below stop.least or not finite, and a slot that has stopped writes -1.
template <int T>
__global__ void __launch_bounds__(T)
k_reduce(const double* partial, int count, int groups, double* __restrict__ out, StopRule stop) {
    __shared__ double red[T];
    grid_begin();
    const int slot = blockIdx.x / groups, grp = blockIdx.x % groups;
    const bool live = !stop.flags || (stop.flags[slot] & SF_ACTIVE);
    if (!live) {   // uniform over the CTA
        if (threadIdx.x == 0) out[blockIdx.x] = -1.0;
        return;
    }
    const int per = count / groups;
    const double* p = partial + (long long)slot * count + (long long)grp * per;
    double acc = 0.0;
    for (int i = threadIdx.x; i < per; i += T) acc += p[i];
    const double s = block_sum<T>(acc, red);
    if (threadIdx.x != 0) return;
    out[blockIdx.x] = s;
    if (stop.flags && !(s >= stop.least[slot] && isfinite(s))) stop.flags[slot] = 0;
}

template <typename R>
__global__ void k_init_tau(GridDesc g, unsigned mask, R* __restrict__ tau) {
    const int slot = blockIdx.y;
    if (!slot_active(g, mask, slot)) return;
    R v[3][3];   // (k + k0) E_c of each phase, rounded once
    for (int p = 0; p < 3; ++p)
        for (int c = 0; c < 3; ++c) v[p][c] = R(g.KP[p] * g.E[slot][c]);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < g.N3; i += (long long)gridDim.x * blockDim.x) {
        const int ph = g.phase[i];
        for (int c = 0; c < 3; ++c)
            tau[((long long)slot * 3 + c) * g.N3 + i] = ph == 0 ? v[0][c] : (ph == 1 ? v[1][c] : v[2][c]);
    }
}

template <typename R>
__global__ void k_e_to_tau(GridDesc g, int slot, const double* __restrict__ e, R* __restrict__ tau) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < g.N3; i += (long long)gridDim.x * blockDim.x) {
        const int ph = g.phase[i];
        const double kp = ph == 0 ? g.KP[0] : (ph == 1 ? g.KP[1] : g.KP[2]);
        for (int c = 0; c < 3; ++c) tau[((long long)slot * 3 + c) * g.N3 + i] = R(kp * e[c * g.N3 + i]);
    }
}

// e = tau / (k + k0).  The three divisors are known, so each quotient is a product with the
// reciprocal in two parts (Brisebarre, Muller & Raina, "Accelerating correctly rounded
// floating-point division when the divisor is known in advance", 2004), which is within one unit
// in the last place, and one residual step with the rounded reciprocal, which then rounds
// correctly for every divisor (Markstein, "Computation of elementary functions on the IBM RISC
// System/6000 processor", 1990): four FP64 operations instead of a divide's ten or so, which bound
// this kernel.  Operands whose residual could leave the normal range are divided.  The reciprocals
// come from the host: formed in every thread they cost more FP64 operations than the one or two
// voxels that a thread of a grid up to 96^3 has (a call of one FP32 sweep at 96^3 142 -> 117 us).
struct Reciprocals {
    double rc[3], rl[3];   // 1 / KP = rc + rl
};

template <typename R>
__global__ void k_tau_to_e(GridDesc g, Reciprocals kr, int slot, const R* __restrict__ tau, double* __restrict__ e) {
    auto in_range = [](double d) {   // 2^-823 <= |d| < 2^777, without the FP64 pipe
        return ((unsigned)__double2hiint(d) >> 20 & 0x7ffu) - 200u < 1600u;
    };
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < g.N3; i += (long long)gridDim.x * blockDim.x) {
        const int ph = g.phase[i];
        const double kp = ph == 0 ? g.KP[0] : (ph == 1 ? g.KP[1] : g.KP[2]);
        const double r = ph == 0 ? kr.rc[0] : (ph == 1 ? kr.rc[1] : kr.rc[2]);
        const double l = ph == 0 ? kr.rl[0] : (ph == 1 ? kr.rl[1] : kr.rl[2]);
        for (int c = 0; c < 3; ++c) {
            const double t = (double)tau[((long long)slot * 3 + c) * g.N3 + i];
            const double q = fma(t, r, t * l);
            double v = fma(fma(-q, kp, t), r, q);
            if (!(in_range(t) && in_range(q))) v = t == 0.0 ? t : t / kp;
            e[c * g.N3 + i] = v;
        }
    }
}

__global__ void k_widen(GridDesc g, unsigned mask, const float* __restrict__ src, double* __restrict__ dst) {
    const int slot = blockIdx.y;
    if (!slot_active(g, mask, slot)) return;
    const long long n = 3 * g.N3, off = (long long)slot * n;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[off + i] = (double)src[off + i];
}

__global__ void k_axpy(GridDesc g, unsigned mask, const float* __restrict__ d, double* __restrict__ tau) {
    const int slot = blockIdx.y;
    if (!slot_active(g, mask, slot)) return;
    const long long n = 3 * g.N3, off = (long long)slot * n;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        tau[off + i] += (double)d[off + i];
}

template <typename R>
__global__ void k_convert(const double* __restrict__ s, R* __restrict__ d, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        d[i] = R(s[i]);
}

template <typename R>
__global__ void k_convert_back(const R* __restrict__ s, double* __restrict__ d, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        d[i] = (double)s[i];
}

// ---------------------------------------------------------------------------
// launch wrappers
// ---------------------------------------------------------------------------

static int pointwise_blocks(long long n) {
    long long b = (n + kThreads - 1) / kThreads;
    return (int)(b < 152 * 16 ? b : 152 * 16);
}

template <> int x_ctas_for<float>(const GridDesc& g) {
    if (g.xyvar == 1 && fused_cluster(g.N)) return fused_xy_ctas(g);
    const int f = fast_x_ctas(g);
    return f ? f : gen_x_ctas(g);
}
template <> int x_ctas_for<double>(const GridDesc& g) { return fx_x_ctas(g); }
template <> int z_ctas_for<float>(const GridDesc& g) {
    const int f = fast_z_ctas(g);
    return f ? f : gen_z_ctas(g);
}
template <> int z_ctas_for<double>(const GridDesc& g) { return fx_z_ctas(g); }

// FP64: block fixed point.  FP32: the kernels of hmg_fast.cu for N = 64, 96, 128, 192, 256 and
// 512, those of hmg_gen32.cu for every other size.
template <typename R>
void launch_x_forward(const GridDesc& g, int mode, unsigned mask, const R* tau, void* spec,
                      double* partial, cudaStream_t st) {
    if constexpr (std::is_same<R, double>::value) fx_x_forward(g, mode, mask, tau, spec, partial, st);
    else if (!fast_x_forward(g, mode, mask, tau, spec, partial, st)) gen_x_forward(g, mode, mask, tau, spec, partial, st);
}

template <typename R>
void launch_y_pass(const GridDesc& g, bool forward, unsigned mask, void* spec, cudaStream_t st) {
    if constexpr (std::is_same<R, double>::value) fx_y(g, forward, mask, spec, st);
    else if (!fast_y(g, forward, mask, spec, st)) gen_col(g, false, forward, mask, spec, st);
}

template <typename R>
void launch_z_pass(const GridDesc& g, int mode, unsigned mask, void* spec, double* partial, cudaStream_t st) {
    if constexpr (std::is_same<R, double>::value) {
        if (mode == Z_FWD) fx_z_plain(g, true, mask, spec, spec, st);
        else fx_z(g, mode, mask, spec, partial, st);
    } else if (!fast_z(g, mode, mask, spec, partial, st)) {
        gen_z(g, mode, mask, spec, partial, st);
    }
}

void launch_z_inverse_from(const GridDesc& g, unsigned mask, const void* src, void* spec, cudaStream_t st) {
    fx_z_plain(g, false, mask, src, spec, st);
}

template <typename R>
void launch_x_inverse(const GridDesc& g, int mode, unsigned mask, const void* spec, R* tau,
                      const float* r32, float* d32, float* r32_out, double* partial, cudaStream_t st) {
    if constexpr (std::is_same<R, double>::value) fx_x_inverse(g, mode, mask, spec, tau, d32, r32_out, partial, st);
    else if (!fast_x_inverse(g, mode, mask, spec, tau, r32, partial, st)) gen_x_inverse(g, mode, mask, spec, tau, r32, partial, st);
}

template <typename R>
bool launch_xy_forward(const GridDesc& g, int mode, unsigned mask, const R* tau, void* spec, double* partial,
                       cudaStream_t st) {
    if constexpr (std::is_same<R, float>::value) {
        if (g.xyvar == 1 && fused_xy_forward(g, mode, mask, tau, spec, partial, st)) return true;
    }
    launch_x_forward<R>(g, mode, mask, tau, spec, partial, st);
    launch_y_pass<R>(g, true, mask, spec, st);
    return false;
}

template <typename R>
bool launch_yx_inverse(const GridDesc& g, int mode, unsigned mask, const void* spec, R* tau, const float* r32,
                       float* d32, float* r32_out, double* partial, cudaStream_t st) {
    if constexpr (std::is_same<R, float>::value) {
        if (g.xyvar == 1 && fused_yx_inverse(g, mode, mask, spec, tau, r32, partial, st)) return true;
    }
    launch_y_pass<R>(g, false, mask, const_cast<void*>(spec), st);
    launch_x_inverse<R>(g, mode, mask, spec, tau, r32, d32, r32_out, partial, st);
    return false;
}

void launch_reduce(const double* partial, int nslots, int count, int groups, double* out, cudaStream_t st,
                   const StopRule& stop) {
    const dim3 grid(nslots * groups);
    if (count / groups > 4096) launch_kernel(true, k_reduce<1024>, grid, 1024, 0, st, partial, count, groups, out, stop);
    else launch_kernel(true, k_reduce<256>, grid, 256, 0, st, partial, count, groups, out, stop);
}

template <typename R>
void launch_init_tau(const GridDesc& g, unsigned mask, R* tau, cudaStream_t st) {
    k_init_tau<R><<<dim3(pointwise_blocks(g.N3), g.nslots), kThreads, 0, st>>>(g, mask, tau);
}
template <typename R>
void launch_e_to_tau(const GridDesc& g, int slot, const double* e, R* tau, cudaStream_t st) {
    k_e_to_tau<R><<<pointwise_blocks(g.N3), kThreads, 0, st>>>(g, slot, e, tau);
}
template <typename R>
void launch_tau_to_e(const GridDesc& g, int slot, const R* tau, double* e, cudaStream_t st) {
    Reciprocals kr;
    for (int p = 0; p < 3; ++p) {
        kr.rc[p] = 1.0 / g.KP[p];
        kr.rl[p] = std::fma(-kr.rc[p], g.KP[p], 1.0) * kr.rc[p];
    }
    k_tau_to_e<R><<<pointwise_blocks(g.N3), kThreads, 0, st>>>(g, kr, slot, tau, e);
}
void launch_widen(const GridDesc& g, unsigned mask, const float* src, double* dst, cudaStream_t st) {
    k_widen<<<dim3(pointwise_blocks(3 * g.N3), g.nslots), kThreads, 0, st>>>(g, mask, src, dst);
}
void launch_axpy(const GridDesc& g, unsigned mask, const float* d, double* tau, cudaStream_t st) {
    k_axpy<<<dim3(pointwise_blocks(3 * g.N3), g.nslots), kThreads, 0, st>>>(g, mask, d, tau);
}
template <typename R>
void launch_convert(const double* src, R* dst, long long n, cudaStream_t st) {
    k_convert<R><<<pointwise_blocks(n), kThreads, 0, st>>>(src, dst, n);
}
template <typename R>
void launch_convert_back(const R* src, double* dst, long long n, cudaStream_t st) {
    k_convert_back<R><<<pointwise_blocks(n), kThreads, 0, st>>>(src, dst, n);
}

#define HMG_INST(R)                                                                                         \
    template void launch_x_forward<R>(const GridDesc&, int, unsigned, const R*, void*, double*, cudaStream_t); \
    template void launch_y_pass<R>(const GridDesc&, bool, unsigned, void*, cudaStream_t);                   \
    template void launch_z_pass<R>(const GridDesc&, int, unsigned, void*, double*, cudaStream_t);           \
    template void launch_x_inverse<R>(const GridDesc&, int, unsigned, const void*, R*, const float*, float*, \
                                      float*, double*, cudaStream_t);                                       \
    template void launch_init_tau<R>(const GridDesc&, unsigned, R*, cudaStream_t);                          \
    template bool launch_xy_forward<R>(const GridDesc&, int, unsigned, const R*, void*, double*, cudaStream_t); \
    template bool launch_yx_inverse<R>(const GridDesc&, int, unsigned, const void*, R*, const float*, float*,   \
                                       float*, double*, cudaStream_t);                                        \
    template void launch_e_to_tau<R>(const GridDesc&, int, const double*, R*, cudaStream_t);                \
    template void launch_tau_to_e<R>(const GridDesc&, int, const R*, double*, cudaStream_t);                \
    template void launch_convert<R>(const double*, R*, long long, cudaStream_t);                            \
    template void launch_convert_back<R>(const R*, double*, long long, cudaStream_t);
HMG_INST(float)
HMG_INST(double)
#undef HMG_INST

}  // namespace hmg
