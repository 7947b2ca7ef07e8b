// FP32 pass kernels for the grid sizes without the kernels of hmg_fast.cu (N = 8 .. 54, 72,
// 108, 144, 162, 216, 288, 324, 384, 432, 486).
//
// One 1D transform is two radix stages in registers with one shared-memory exchange (three
// stages for lengths 243 and 486), all sizes known at compile time.  The shared-memory
// Stockham kernels these replace took each stage through memory with run-time divisions for
// every index, at a sixth to a tenth of the copy bandwidth; here an x, y or z pass is bound by
// the instructions of its addressing and by latency (y by HBM).  144^3, three gradients, us
// per launch, before and now: x forward 152 and 55, y 143 and 37, z 227 and 62; x inverse
// plus x forward 369, chained 98.
// The passes, layouts and float operations per voxel are those described in hmg_kernels.cu;
// the chained x round trip is that of hmg_fast.cu.
#pragma once

#include "hmg_cta.cuh"
#include "hmg_fft.cuh"
#include "hmg_fixed.cuh"
#include "hmg_green.cuh"
#include "hmg_launch.cuh"

namespace hmg {
namespace g32 {

using fx::Dft;
using fx::mkc;
using fx::PlanOf;
using fx::swap_ri;
using fx::operator+;
using fx::operator-;

// Radices and threads per pencil (hmg_fixed.cuh); FP32 values take half the registers of the
// fixed-point ones, so two long stages are the better split here.
template <int L> struct Plan;
template <> struct Plan<4> : PlanOf<4, 1, 1, 1> {};
template <> struct Plan<6> : PlanOf<6, 1, 1, 1> {};
template <> struct Plan<8> : PlanOf<8, 1, 1, 1> {};
template <> struct Plan<9> : PlanOf<9, 1, 1, 1> {};
template <> struct Plan<12> : PlanOf<4, 3, 1, 4> {};
template <> struct Plan<16> : PlanOf<4, 4, 1, 4> {};
template <> struct Plan<18> : PlanOf<6, 3, 1, 6> {};
template <> struct Plan<24> : PlanOf<6, 4, 1, 6> {};
template <> struct Plan<27> : PlanOf<9, 3, 1, 9> {};
template <> struct Plan<32> : PlanOf<8, 4, 1, 8> {};
template <> struct Plan<36> : PlanOf<6, 6, 1, 6> {};
template <> struct Plan<48> : PlanOf<8, 6, 1, 8> {};
template <> struct Plan<54> : PlanOf<9, 6, 1, 9> {};
template <> struct Plan<72> : PlanOf<9, 8, 1, 9> {};
template <> struct Plan<81> : PlanOf<9, 9, 1, 9> {};
template <> struct Plan<108> : PlanOf<12, 9, 1, 12> {};
template <> struct Plan<144> : PlanOf<12, 12, 1, 12> {};
template <> struct Plan<162> : PlanOf<18, 9, 1, 9> {};
template <> struct Plan<192> : PlanOf<16, 12, 1, 16> {};
template <> struct Plan<216> : PlanOf<18, 12, 1, 18> {};
template <> struct Plan<243> : PlanOf<9, 9, 3, 27> {};
template <> struct Plan<288> : PlanOf<18, 16, 1, 18> {};
template <> struct Plan<324> : PlanOf<18, 18, 1, 18> {};
template <> struct Plan<384> : PlanOf<24, 16, 1, 24> {};
template <> struct Plan<432> : PlanOf<24, 18, 1, 24> {};
template <> struct Plan<486> : PlanOf<9, 9, 6, 54> {};

// CTAs of about 128 to 256 threads; columns in runs of up to 16 (128 bytes)
template <int M> constexpr int x_rows() { return divisor_upto(4LL * M * M, 160 / Plan<M>::TPP > 1 ? 160 / Plan<M>::TPP : 1); }
template <int L> constexpr int col_cols() {
    const int lim = 256 / Plan<L>::TPP;
    return divisor_upto(L / 2, lim < 4 ? 4 : lim > 16 ? 16 : lim);
}
template <int L> constexpr int z_cols() {
    const int lim = 288 / (3 * Plan<L>::TPP);
    return divisor_upto(L / 2, lim < 4 ? 4 : lim > 8 ? 8 : lim);
}
// registers: 64 per thread, 80 where a thread holds 24 values
template <int L> constexpr int min_ctas(int threads) {
    const int t = (threads + 31) / 32 * 32, per = Plan<L>::R0 > 18 ? 768 : 1024;
    return t >= per ? 1 : per / t;
}

// ---------------------------------------------------------------------------
// forward transform of one pencil (see fx::transform)
// ---------------------------------------------------------------------------
template <int L, int R, int NSP, int IT, class S>
__device__ __forceinline__ void stage_read(float2 (&v)[IT][R], int t, int pen, const float2* sm,
                                           const float2* __restrict__ tw) {
    constexpr int TPP = Plan<L>::TPP, J = L / R, TS = L / (NSP * R);
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int j = t + it * TPP;
        if (J % TPP == 0 || j < J) {
            const int k = j % NSP;
#pragma unroll
            for (int r = 0; r < R; ++r) v[it][r] = sm[S::at(j + r * J, pen)];
#pragma unroll
            for (int r = 1; r < R; ++r) v[it][r] = cmul(v[it][r], __ldg(&tw[k * r * TS]));
            Dft<R>::run(v[it]);
        }
    }
}
template <int L, int R, int NSP, int IT, class F>
__device__ __forceinline__ void stage_emit(const float2 (&v)[IT][R], int t, F f) {
    constexpr int TPP = Plan<L>::TPP, J = L / R;
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int j = t + it * TPP;
        if (J % TPP == 0 || j < J) {
            const int base = (j / NSP) * NSP * R + j % NSP;
#pragma unroll
            for (int r = 0; r < R; ++r) f(base + r * NSP, v[it][r], it, r);
        }
    }
}
// first-stage inputs of this thread: f(index) -> value
template <int L, class F>
__device__ __forceinline__ void first_fill(float2 (&v)[Plan<L>::I0][Plan<L>::R0], int t, F f) {
    using P = Plan<L>;
    constexpr int J = L / P::R0;
#pragma unroll
    for (int it = 0; it < P::I0; ++it) {
        const int j = t + it * P::TPP;
        if (J % P::TPP == 0 || j < J) {
#pragma unroll
            for (int r = 0; r < P::R0; ++r) v[it][r] = f(j + r * J);
        }
    }
}
template <int L, class S>
__device__ __forceinline__ void transform(float2 (&v)[Plan<L>::I0][Plan<L>::R0], float2 (&o)[Plan<L>::IL][Plan<L>::RL],
                                          int t, int pen, float2* sm, const float2* __restrict__ tw) {
    using P = Plan<L>;
#pragma unroll
    for (int it = 0; it < P::I0; ++it)
        if ((L / P::R0) % P::TPP == 0 || t + it * P::TPP < L / P::R0) Dft<P::R0>::run(v[it]);
    if constexpr (P::NS == 1) {
#pragma unroll
        for (int r = 0; r < P::R0; ++r) o[0][r] = v[0][r];
    } else {
        stage_emit<L, P::R0, 1, P::I0>(v, t, [&](int k, float2 z, int, int) { sm[S::at(k, pen)] = z; });
        __syncthreads();
        if constexpr (P::NS == 2) {
            stage_read<L, P::R1, P::R0, P::I1, S>(o, t, pen, sm, tw);
        } else {
            float2 u[P::I1][P::R1];
            stage_read<L, P::R1, P::R0, P::I1, S>(u, t, pen, sm, tw);
            __syncthreads();   // every thread has read the previous stage
            stage_emit<L, P::R1, P::R0, P::I1>(u, t, [&](int k, float2 z, int, int) { sm[S::at(k, pen)] = z; });
            __syncthreads();
            stage_read<L, P::R2, P::R0 * P::R1, P::I2, S>(o, t, pen, sm, tw);
        }
    }
}
template <int L, class F>
__device__ __forceinline__ void last_emit(const float2 (&o)[Plan<L>::IL][Plan<L>::RL], int t, F f) {
    stage_emit<L, Plan<L>::RL, Plan<L>::NL, Plan<L>::IL>(o, t, f);
}

// Shared-memory slots of rows (padded where the first radix is even) and columns, as Slots in
// hmg_fixed.cuh.
template <int L, int NPEN>
struct RowSlots {
    static constexpr int PAD = Plan<L>::R0 % 2 == 0 ? Plan<L>::R0 : 0;
    static constexpr int LEN = PAD ? L + L / PAD : L;
    static constexpr int TOTAL = LEN * NPEN;
    HMG_HD static int at(int i, int pen) { return pen * LEN + (PAD ? i + i / (PAD ? PAD : 1) : i); }
};
template <int NPEN>
struct ColSlots {
    HMG_HD static int at(int i, int pen) { return i * NPEN + pen; }
};

// ---------------------------------------------------------------------------
// x passes
// ---------------------------------------------------------------------------
template <int M>
struct XShape {
    static constexpr int N = 2 * M, RW = x_rows<M>(), TPP = Plan<M>::TPP, T = RW * TPP;
    using S = RowSlots<M, RW>;
    static constexpr size_t smem = sizeof(float2) * S::TOTAL;
};

struct Coef {
    float c0, c1, c2;
    __device__ float at(int ph) const { return ph == 0 ? c0 : (ph == 1 ? c1 : c2); }
    __device__ float2 at(uchar2 q) const { return make_float2(at(q.x), at(q.y)); }
};

// Real split of the row transform held in o, through shared memory, written to dst:
// X_k = e + o w_N^k with e = (Z_k + conj Z_{M-k}) / 2, o = -i (Z_k - conj Z_{M-k}) / 2; X_0 packs
// X(0) and X(N/2).  The buffer is free again after the caller's next barrier.
template <int M>
__device__ __forceinline__ void split_store(const float2 (&o)[Plan<M>::IL][Plan<M>::RL], int t, int r, float2* sm,
                                            const float2* __restrict__ twN, float2* __restrict__ dst) {
    using S = typename XShape<M>::S;
    if (Plan<M>::NS > 1) __syncthreads();   // the last stage has been read by every thread
    last_emit<M>(o, t, [&](int k, float2 z, int, int) { sm[S::at(k, r)] = z; });
    __syncthreads();
    for (int k = t; k < M; k += Plan<M>::TPP) {
        const float2 z = sm[S::at(k, r)];
        float2 out;
        if (k == 0) {
            out = make_float2(z.x + z.y, z.x - z.y);
        } else {
            const float2 zm = sm[S::at(M - k, r)];
            const float2 e = make_float2(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y));
            const float2 d = make_float2(0.5f * (z.y + zm.y), -0.5f * (z.x - zm.x));
            out = e + cmul(d, __ldg(&twN[k]));
        }
        dst[k] = out;
    }
}
// Complex-to-real merge of a row spectrum into the first stage (swapped for the inverse):
// (X_k + conj X_{M-k}) + i w_N^-k (X_k - conj X_{M-k}).
template <int M>
__device__ __forceinline__ void merge_load(float2 (&v)[Plan<M>::I0][Plan<M>::R0], int t, const float2* src,
                                           const float2* __restrict__ twN) {
    first_fill<M>(v, t, [&](int k) {
        float2 a = src[k], b = src[k ? M - k : 0];
        if (k == 0) {   // packed X(0) + i X(N/2)
            b = make_float2(a.y, 0.f);
            a = make_float2(a.x, 0.f);
        }
        const float2 s = make_float2(a.x + b.x, a.y - b.y), d = make_float2(a.x - b.x, a.y + b.y);
        const float2 dw = cmulc(d, __ldg(&twN[k]));
        return make_float2(s.y + dw.x, s.x - dw.y);
    });
}

// (double)f by moving its bits: the conversion instruction shares the FP64 pipe (2 per clock and
// SM), which bounds the residual sweep; only subnormals, infinities and NaN use it.
__device__ __forceinline__ double widen(float f) {
    const unsigned u = __float_as_uint(f), e = u >> 23 & 0xffu;
    if (e - 1u >= 254u) return f == 0.f ? 0.0 : (double)f;
    return __hiloint2double((int)((u & 0x80000000u) | ((u & 0x7fffffffu) >> 3) + 0x38000000u), (int)(u << 29));
}

template <int M, int MODE>
__global__ void __launch_bounds__(XShape<M>::T, min_ctas<M>(XShape<M>::T))
k_gx_forward(GridDesc g, unsigned mask, const float* tau, float2* __restrict__ spec,
             double* __restrict__ partial) {
    using X = XShape<M>;
    using P = Plan<M>;
    constexpr int N = X::N, RW = X::RW, T = X::T;
    grid_begin();
    const int slot = blockIdx.y;
    if (!slot_active(g, mask, slot)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* sm = reinterpret_cast<float2*>(smem_raw);
    const int r = threadIdx.x / X::TPP, t = threadIdx.x % X::TPP;
    const long long rs = (long long)blockIdx.x * RW + r;                     // c, z, y
    const long long row = (long long)slot * 3 * N * N + rs;
    const float2* src = reinterpret_cast<const float2*>(tau) + row * M;
    const uchar2* ph = reinterpret_cast<const uchar2*>(g.phase) + rs % ((long long)N * N) * M;
    const Coef cf = MODE == XF_FLUX ? Coef{(float)g.W[0], (float)g.W[1], (float)g.W[2]}
                                    : Coef{(float)g.Y[0], (float)g.Y[1], (float)g.Y[2]};
    float2 v[P::I0][P::R0], o[P::IL][P::RL];
    double acc = 0.0;
    first_fill<M>(v, t, [&](int k) {
        float2 d = src[k];
        if (MODE != XF_PLAIN) {
            d = __fmul2_rn(d, cf.at(ph[k]));   // rounded products, as in the chained form
            if (MODE == XF_FLUX) acc += widen(d.x) + widen(d.y);
        }
        return d;
    });
    transform<M, typename X::S>(v, o, t, r, sm, g.tw32 + N);
    split_store<M>(o, t, r, sm, g.tw32, spec + row * M);
    if (MODE == XF_FLUX) {
        __shared__ double red[pow2_at_least(T)];
        const double s = cta_sum<T>(acc, red);
        if (threadIdx.x == 0) partial[(long long)slot * gridDim.x + blockIdx.x] = s;
    }
}

template <int M, bool RES>
__global__ void __launch_bounds__(XShape<M>::T, min_ctas<M>(XShape<M>::T))
k_gx_inverse(GridDesc g, unsigned mask, int mode, const float2* spec, float* __restrict__ tau,
             const float* r32, double* __restrict__ partial) {
    using X = XShape<M>;
    using P = Plan<M>;
    constexpr int N = X::N, RW = X::RW, T = X::T;
    grid_begin();
    const int slot = blockIdx.y;
    if (!slot_active(g, mask, slot)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* sm = reinterpret_cast<float2*>(smem_raw);
    const int r = threadIdx.x / X::TPP, t = threadIdx.x % X::TPP;
    const long long row = (long long)slot * 3 * N * N + (long long)blockIdx.x * RW + r;
    float2 v[P::I0][P::R0], o[P::IL][P::RL];
    merge_load<M>(v, t, spec + row * M, g.tw32);
    transform<M, typename X::S>(v, o, t, r, sm, g.tw32 + N);
    // output step: relaxation, r of the correction sweeps, residual against the old field
    const bool kadd = mode == XI_ADD_R || mode == XI_ADD_R_RES;
    const bool res = RES && (g.dflags ? g.resid != 0 : true);
    const bool addr = kadd && (g.dflags ? (g.dflags[slot] & SF_ADDR) != 0 : true);
    const bool relax = g.relax != 0.0;
    const float wn = (float)(1.0 - g.relax), wo = (float)g.relax;
    float2* out = reinterpret_cast<float2*>(tau) + row * M;
    const float2* rin = reinterpret_cast<const float2*>(r32) + row * M;
    double acc = 0.0;
    last_emit<M>(o, t, [&](int k, float2 z, int, int) {
        float2 n = swap_ri(z), old = make_float2(0.f, 0.f);
        if (res || relax) old = out[k];
        if (relax) n = make_float2(wn * n.x + wo * old.x, wn * n.y + wo * old.y);
        if (addr) {
            const float2 q = rin[k];
            n = make_float2(__fadd_rn(n.x, q.x), __fadd_rn(n.y, q.y));
        }
        if (res) {
            const double da = widen(n.x) - widen(old.x), db = widen(n.y) - widen(old.y);
            acc += da * da;
            acc += db * db;
        }
        out[k] = n;
    });
    if (RES) {   // uniform across the CTA
        __shared__ double red[pow2_at_least(T)];
        const double s = cta_sum<T>(acc, red);
        if (threadIdx.x == 0 && res) partial[(long long)slot * gridDim.x + blockIdx.x] = s;
    }
}

// x inverse of one sweep, update, polarization and x forward of the next, in place (the
// chained form of hmg_fast.cu's k_fx_round); same float operations as the two passes.
template <int M>
__global__ void __launch_bounds__(XShape<M>::T, min_ctas<M>(XShape<M>::T))
k_gx_round(GridDesc g, unsigned mask, int add, int wtau, float2* __restrict__ spec, float* __restrict__ tau,
           const float* r32) {
    using X = XShape<M>;
    using P = Plan<M>;
    using S = typename X::S;
    constexpr int N = X::N, RW = X::RW;
    grid_begin();
    const int slot = blockIdx.y;
    if (!slot_active(g, mask, slot)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* sm = reinterpret_cast<float2*>(smem_raw);
    const int r = threadIdx.x / X::TPP, t = threadIdx.x % X::TPP;
    const long long rs = (long long)blockIdx.x * RW + r;                     // c, z, y
    const long long row = (long long)slot * 3 * N * N + rs;
    const uchar2* ph = reinterpret_cast<const uchar2*>(g.phase) + rs % ((long long)N * N) * M;
    const Coef cf{(float)g.Y[0], (float)g.Y[1], (float)g.Y[2]};
    const bool addr = add && (g.dflags ? (g.dflags[slot] & SF_ADDR) != 0 : true);
    float2 v[P::I0][P::R0], o[P::IL][P::RL];
    merge_load<M>(v, t, spec + row * M, g.tw32);
    transform<M, S>(v, o, t, r, sm, g.tw32 + N);
    float2* out = reinterpret_cast<float2*>(tau) + row * M;
    const float2* rin = reinterpret_cast<const float2*>(r32) + row * M;
    // the last stage's positions are the first stage's where the plan is symmetric
    constexpr bool kSame = P::RL == P::R0;
    if (P::NS > 1 && !kSame) __syncthreads();   // the last stage has been read by every thread
    last_emit<M>(o, t, [&](int k, float2 z, int it, int q) {
        float2 n = swap_ri(z);
        if (addr) {
            const float2 d = rin[k];
            n = make_float2(__fadd_rn(n.x, d.x), __fadd_rn(n.y, d.y));
        }
        if (wtau) out[k] = n;
        n = __fmul2_rn(n, cf.at(ph[k]));
        if constexpr (kSame) v[it][q] = n;
        else sm[S::at(k, r)] = n;
    });
    __syncthreads();
    if constexpr (!kSame) {
        first_fill<M>(v, t, [&](int k) { return sm[S::at(k, r)]; });
        __syncthreads();
    }
    transform<M, S>(v, o, t, r, sm, g.tw32 + N);
    split_store<M>(o, t, r, sm, g.tw32, spec + row * M);
}

// ---------------------------------------------------------------------------
// columns along y (or z, for a plain transform) of one component, in place
// ---------------------------------------------------------------------------
template <int L>
struct ColShape {
    static constexpr int M = L / 2, NP = col_cols<L>(), TPP = Plan<L>::TPP, T = NP * TPP;
    static constexpr size_t smem = sizeof(float2) * L * NP;
};

template <int L>
__global__ void __launch_bounds__(ColShape<L>::T, min_ctas<L>(ColShape<L>::T))
k_gcol(GridDesc g, unsigned mask, int zdir, int inverse, float2* __restrict__ spec) {
    using C = ColShape<L>;
    using P = Plan<L>;
    constexpr int M = C::M, NP = C::NP;
    grid_begin();
    const int slot = blockIdx.y;
    if (!slot_active(g, mask, slot)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* sm = reinterpret_cast<float2*>(smem_raw);
    const int p = threadIdx.x % NP, t = threadIdx.x / NP;
    const int kx = blockIdx.x % (M / NP) * NP + p, cw = blockIdx.x / (M / NP);   // c L + z, or c L + ky
    const long long comp = (long long)slot * 3 + cw / L;
    float2* base = spec + (zdir ? comp * L * L * M + (long long)(cw % L) * M : ((long long)slot * 3 * L + cw) * L * M) + kx;
    const long long step = zdir ? (long long)L * M : M;
    float2 v[P::I0][P::R0], o[P::IL][P::RL];
    if (inverse) first_fill<L>(v, t, [&](int i) { return swap_ri(base[i * step]); });
    else first_fill<L>(v, t, [&](int i) { return base[i * step]; });
    transform<L, ColSlots<NP>>(v, o, t, p, sm, g.tw32);
    if (inverse) last_emit<L>(o, t, [&](int k, float2 z, int, int) { base[k * step] = swap_ri(z); });
    else last_emit<L>(o, t, [&](int k, float2 z, int, int) { base[k * step] = z; });
}

// ---------------------------------------------------------------------------
// z pass of a sweep (Z_ITER, Z_ITER_NOB) or an equilibrium test (Z_EQ)
// ---------------------------------------------------------------------------
template <int L>
struct ZShape {
    static constexpr int M = L / 2, NP = z_cols<L>(), P3 = 3 * NP, TPP = Plan<L>::TPP, T = P3 * TPP;
    static constexpr size_t smem = sizeof(float2) * L * P3;
};

template <int L>
__global__ void __launch_bounds__(ZShape<L>::T, min_ctas<L>(ZShape<L>::T))
k_gz(GridDesc g, unsigned mask, int mode, float2* __restrict__ spec, double* __restrict__ partial) {
    using Z = ZShape<L>;
    using P = Plan<L>;
    using S = ColSlots<Z::P3>;
    constexpr int N = L, M = Z::M, NP = Z::NP, P3 = Z::P3, T = Z::T;
    grid_begin();
    const int slot = blockIdx.y;
    if (!slot_active(g, mask, slot)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* sm = reinterpret_cast<float2*>(smem_raw);
    const int cp = threadIdx.x % P3, t = threadIdx.x / P3;
    const int kx0 = blockIdx.x % (M / NP) * NP, ky = blockIdx.x / (M / NP);
    float2* base = spec + ((long long)slot * 3 + cp / NP) * L * L * M + (long long)ky * M + kx0 + cp % NP;
    constexpr long long step = (long long)L * M;
    float2 v[P::I0][P::R0], o[P::IL][P::RL];
    first_fill<L>(v, t, [&](int i) { return base[i * step]; });
    transform<L, S>(v, o, t, cp, sm, g.tw32);
    if (P::NS > 1) __syncthreads();   // the last stage has been read by every thread
    last_emit<L>(o, t, [&](int k, float2 z, int, int) { sm[S::at(k, cp)] = z; });
    __syncthreads();
    if (mode == Z_EQ) {
        double acc = 0.0;
        for (int q = threadIdx.x; q < L * NP; q += T) {
            const float2* m = sm + q / NP * P3 + q % NP;
            acc += eq_mode(kx0 + q % NP, ky, q / NP, N, m[0], m[NP], m[2 * NP]);
        }
        __syncthreads();   // sm is free: the sum reuses it
        const double twopi_n = 6.283185307179586476925 / (double)N;
        const double s = cta_sum<T>(acc, reinterpret_cast<double*>(smem_raw)) * twopi_n * twopi_n /
                         ((double)g.N3 * (double)g.N3);
        if (threadIdx.x == 0) partial[(long long)slot * gridDim.x + blockIdx.x] = s;
        return;
    }
    const bool addb = g.dflags ? (g.dflags[slot] & SF_ADDB) != 0 : mode == Z_ITER;
    const float scale = (float)(1.0 / (double)g.N3), ga = (float)g.ga, gb = (float)g.gb;
    const float cE[3] = {(float)(g.gc * g.E[slot][0]), (float)(g.gc * g.E[slot][1]), (float)(g.gc * g.E[slot][2])};
    for (int q = threadIdx.x; q < L * NP; q += T) {
        float2* m = sm + q / NP * P3 + q % NP;
        float2 s0 = m[0], s1 = m[NP], s2 = m[2 * NP];
        green_mode_fast<true>(kx0 + q % NP, ky, q / NP, N, scale, ga, gb, addb, cE, s0, s1, s2);
        m[0] = s0;
        m[NP] = s1;
        m[2 * NP] = s2;
    }
    __syncthreads();
    first_fill<L>(v, t, [&](int i) { return swap_ri(sm[S::at(i, cp)]); });
    __syncthreads();
    transform<L, S>(v, o, t, cp, sm, g.tw32);
    last_emit<L>(o, t, [&](int k, float2 z, int, int) { base[k * step] = swap_ri(z); });
}

}  // namespace g32
}  // namespace hmg
