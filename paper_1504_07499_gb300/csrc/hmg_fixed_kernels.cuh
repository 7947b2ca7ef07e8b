// FP64 pass kernels in block fixed point (see hmg_fixed.cuh for the number format).
//
// The sweep has the structure of hmg_kernels.cu: x forward, y forward, z forward + Green
// operator + z inverse, y inverse, x inverse.  The spectrum between the passes is c64
// integers in the packed layout, and each value's exponent belongs to the pencil that wrote
// it: expA holds one per x row [slot][c][z][y] (x forward) or per z column [slot][c][ky][kx]
// (z pass), expB one per y column [slot][c][z][kx] (y passes).
//
// What bounds them (256^3, one gradient): the IMAD.WIDE pipe (16 per clock and SM; 24 per
// value in a column pass, 59 in the z pass, whose 0.54 ms it could do in 0.32), then latency;
// FP64 is left for the coefficient product, the flux sum and the residual (1 to 2 operations
// per real value).  Against the FP64 butterflies these replace, one sweep of one gradient
// at 256^3 through the C ABI went 9.7 -> 1.8 ms (copies and conversions of the field included).
#pragma once

#include "hmg_cta.cuh"
#include "hmg_fft.cuh"
#include "hmg_fixed.cuh"
#include "hmg_green.cuh"
#include "hmg_launch.cuh"

namespace hmg {
namespace fx {

// rows per CTA of an x pass of length M, columns per CTA of a column / z pass of length L:
// about 128 to 256 threads; columns in runs of at least 64 bytes where N/2 allows it
template <int M> constexpr int x_rows() { return divisor_upto(4LL * M * M, 192 / Plan<M>::TPP > 1 ? 192 / Plan<M>::TPP : 1); }
template <int L> constexpr int col_cols() {
    int lim = 256 / Plan<L>::TPP;
    lim = lim < 4 ? 4 : lim > 16 ? 16 : lim;
    return divisor_upto(L / 2, lim);
}
template <int L> constexpr int z_cols() {
    int lim = 400 / (3 * Plan<L>::TPP);
    lim = lim < 2 ? 2 : lim > 8 ? 8 : lim;
    return divisor_upto(L / 2, lim);
}
// Registers per thread by the threads an SM is to hold: 64 for the column and z passes, 72 to
// 80 for the x passes (64 spill there: x inverse at 192^3 371 us against 197 us).
constexpr int min_ctas(int threads, int per_sm) {
    const int t = (threads + 31) / 32 * 32;
    return t >= per_sm ? 1 : per_sm / t;
}

__device__ __forceinline__ double coef3(int ph, const double* c) { return ph == 0 ? c[0] : (ph == 1 ? c[1] : c[2]); }

// ---------------------------------------------------------------------------
// x forward: FP64 field rows -> packed integer spectrum rows
// ---------------------------------------------------------------------------
template <int M>
struct XShape {
    static constexpr int N = 2 * M, RW = x_rows<M>(), TPP = Plan<M>::TPP, T = RW * TPP;
    using S = Slots<M, RW, true>;
    static constexpr size_t smem = sizeof(c64) * S::TOTAL;
};

// Real split of a row transform (exponent e, scaled from values below 2^E) through shared memory
// and its store to dst; om: one zeroed word per row.
template <int M>
__device__ __forceinline__ void split_store(const GridDesc& g, const c64 (&o)[Plan<M>::IL][Plan<M>::RL], int t, int r,
                                            long long row, c64* dst, c64* sm, unsigned* om, int E, int e) {
    using P = Plan<M>;
    using S = typename XShape<M>::S;
    constexpr int TPP = P::TPP;
    if (P::NS > 1) __syncthreads();   // the last stage has been read by every thread
    unsigned m = 0;
    last_emit<M>(o, t, [&](int k, c64 z) {
        m |= mag(z);
        sm[S::at(k, r)] = z;
    });
    atomicOr(&om[r], m);
    __syncthreads();
    // real split: X_k = (Z_k + conj Z_{M-k} - i w_N^k (Z_k - conj Z_{M-k})) / 2, stored halved
    const int sh = max(0, bits_of(om[r]) - 61);
    e += 1 + sh;
    for (int k = t; k < M; k += TPP) {
        c64 z = sm[S::at(k, r)];
        if (sh) z = shr_round(z, sh);
        c64 out;
        if (k == 0) {
            out = mkc(half(z.x + z.y), half(z.x - z.y));
        } else {
            c64 zm = sm[S::at(M - k, r)];
            if (sh) zm = shr_round(zm, sh);
            const c64 w = cmul4(mkc(z.y + zm.y, zm.x - z.x), __ldg(&g.twf[k]));
            out = quarter(mkc(z.x + zm.x, z.y - zm.y)) + w;
        }
        dst[k] = out;
    }
    if (t == 0) g.expA[row] = exp_is_nan(E) ? kExpNan : e;
}

// Complex-to-real merge of a packed row spectrum into the first stage of the inverse row
// transform (a quarter of it; exponent e); returns whether the row is not a number.  key: one
// word per row, kExpZero.
template <int M>
__device__ __forceinline__ bool load_merge(const GridDesc& g, c64 (&v)[Plan<M>::I0][Plan<M>::R0], int t, int r,
                                           long long row, const c64* src, int* key, int& e) {
    using P = Plan<M>;
    constexpr int TPP = P::TPP, J = M / P::R0;
    const int* ein = g.expB + (long long)((int)row / (2 * M)) * M;   // one exponent per kx of the (slot, c, z) plane
    int mk = kExpZero;
#pragma unroll
    for (int it = 0; it < P::I0; ++it) {
        const int j = t + it * TPP;
        if (J % TPP == 0 || j < J) {
#pragma unroll
            for (int q = 0; q < P::R0; ++q) {
                v[it][q] = src[j + q * J];
                mk = max(mk, ein[j + q * J] + bits_of(mag(v[it][q])));
            }
        }
    }
    atomicMax(&key[r], mk);
    __syncthreads();
    const int E = key[r];
    e = E - first_bits(P::R0);
    // complex-to-real merge, a quarter of it: (X_k + conj X_{M-k}) + i w_N^{-k} (X_k - conj X_{M-k})
#pragma unroll
    for (int it = 0; it < P::I0; ++it) {
        const int j = t + it * TPP;
        if (J % TPP == 0 || j < J) {
#pragma unroll
            for (int q = 0; q < P::R0; ++q) {
                const int k = j + q * J, km = k ? M - k : 0;
                c64 a = shift(v[it][q], ein[k] - e);
                c64 b = shift(src[km], ein[km] - e);
                if (k == 0) {   // packed X(0) + i X(N/2)
                    b = mkc(a.y, 0);
                    a = mkc(a.x, 0);
                }
                const c64 s = quarter(mkc(a.x + b.x, a.y - b.y));
                const c64 d = cmul4(mkc(a.x - b.x, a.y + b.y), conj_tw(__ldg(&g.twf[k])));
                v[it][q] = swap_ri(mkc(s.x - d.y, s.y + d.x));
            }
        }
    }
    e += 2;
    return exp_is_nan(E);
}

template <int M>
__global__ void __launch_bounds__(XShape<M>::T, min_ctas(XShape<M>::T, 896))
k_fxx_forward(GridDesc g, unsigned mask, int mode, const double* tau, c64* __restrict__ spec,
              double* __restrict__ partial) {
    using X = XShape<M>;
    using P = Plan<M>;
    using S = typename X::S;
    constexpr int N = X::N, RW = X::RW, TPP = X::TPP, T = X::T, J = M / P::R0;
    grid_begin();
    const int slot = blockIdx.y;
    if (!slot_active(g, mask, slot)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    c64* sm = reinterpret_cast<c64*>(smem_raw);
    __shared__ int key[RW];
    __shared__ unsigned orm[3 * RW];
    __shared__ double red[pow2_at_least(T)];
    const int r = threadIdx.x / TPP, t = threadIdx.x % TPP;
    for (int i = threadIdx.x; i < 3 * RW; i += T) {
        orm[i] = 0;
        if (i < RW) key[i] = kExpZero;
    }
    const long long row = (long long)slot * 3 * N * N + (long long)blockIdx.x * RW + r;   // slot, c, z, y
    const double2* src = reinterpret_cast<const double2*>(tau) + row * M;
    const uchar2* ph = reinterpret_cast<const uchar2*>(g.phase) + (long long)((int)(blockIdx.x * RW + r) % (N * N)) * M;
    __syncthreads();
    // load, coefficient product (FP64), largest exponent of the row
    c64 v[P::I0][P::R0];
    double acc = 0.0;
    int mk = kExpZero;
    double cf[3];
#pragma unroll
    for (int p = 0; p < 3; ++p) cf[p] = mode == XF_FLUX ? g.W[p] : g.YN[p];
#pragma unroll
    for (int it = 0; it < P::I0; ++it) {
        const int j = t + it * TPP;
        if (J % TPP == 0 || j < J) {
#pragma unroll
            for (int q = 0; q < P::R0; ++q) {
                double2 d = src[j + q * J];
                if (mode != XF_PLAIN) {
                    const uchar2 b = ph[j + q * J];
                    d.x *= coef3(b.x, cf);
                    d.y *= coef3(b.y, cf);
                    if (mode == XF_FLUX) acc += d.x + d.y;
                }
                mk = max(mk, max(key_of(d.x), key_of(d.y)));
                v[it][q] = mkc(__double_as_longlong(d.x), __double_as_longlong(d.y));
            }
        }
    }
    atomicMax(&key[r], mk);
    __syncthreads();
    const int E = key[r];
    int e = E - first_bits(P::R0);
#pragma unroll
    for (int it = 0; it < P::I0; ++it)
        if (J % TPP == 0 || t + it * TPP < J) {
#pragma unroll
            for (int q = 0; q < P::R0; ++q)
                v[it][q] = mkc(to_fixed(__longlong_as_double(v[it][q].x), e), to_fixed(__longlong_as_double(v[it][q].y), e));
        }
    c64 o[P::IL][P::RL];
    transform<M, S>(v, o, t, r, sm, orm, RW, e, g.twf + N);
    split_store<M>(g, o, t, r, row, spec + row * M, sm, orm + 2 * RW, E, e);
    if (mode == XF_FLUX) {
        const double s = cta_sum<T>(acc, red);
        if (threadIdx.x == 0) partial[(long long)slot * gridDim.x + blockIdx.x] = s;
    }
}

// ---------------------------------------------------------------------------
// x inverse: packed integer spectrum rows -> FP64 field rows, with the sweep's output step
// ---------------------------------------------------------------------------
template <int M>
__global__ void __launch_bounds__(XShape<M>::T, min_ctas(XShape<M>::T, 896))
k_fxx_inverse(GridDesc g, unsigned mask, int mode, const c64* spec, double* __restrict__ tau,
              float* __restrict__ d32, float* __restrict__ r32, double* __restrict__ partial) {
    using X = XShape<M>;
    using P = Plan<M>;
    using S = typename X::S;
    constexpr int N = X::N, RW = X::RW, TPP = X::TPP, T = X::T, J = M / P::R0;
    grid_begin();
    const int slot = blockIdx.y;
    if (!slot_active(g, mask, slot)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    c64* sm = reinterpret_cast<c64*>(smem_raw);
    __shared__ int key[RW];
    __shared__ unsigned orm[2 * RW];
    __shared__ double red[pow2_at_least(T)];
    const int r = threadIdx.x / TPP, t = threadIdx.x % TPP;
    for (int i = threadIdx.x; i < 2 * RW; i += T) {
        orm[i] = 0;
        if (i < RW) key[i] = kExpZero;
    }
    const long long row = (long long)slot * 3 * N * N + (long long)blockIdx.x * RW + r;   // slot, c, z, y
    __syncthreads();
    c64 v[P::I0][P::R0];
    int e;
    const bool bad = load_merge<M>(g, v, t, r, row, spec + row * M, key, e);
    c64 o[P::IL][P::RL];
    transform<M, S>(v, o, t, r, sm, orm, RW, e, g.twf + N);
    if (mode != XI_PLAIN) e -= scale_bits(N);
    // output step in FP64
    double2* out = reinterpret_cast<double2*>(tau) + row * M;
    float2* dout = reinterpret_cast<float2*>(d32) + row * M;
    float2* rout = reinterpret_cast<float2*>(r32) + row * M;
    const bool relax = g.relax != 0.0, res = mode == XI_INPLACE_RES || mode == XI_DIFF;
    const double wn = 1.0 - g.relax, wo = g.relax;
    double acc = 0.0;
    auto emit = [&](auto low) {
        last_emit<M>(o, t, [&](int k, c64 z) {
            double2 n = from_fixed<low>(swap_ri(z), e);
            if (bad) n = make_double2(nan(""), nan(""));
            double2 old = make_double2(0.0, 0.0);
            if (res || relax) old = out[k];
            if (relax) n = make_double2(wn * n.x + wo * old.x, wn * n.y + wo * old.y);
            if (res) {
                const double da = n.x - old.x, db = n.y - old.y;
                acc += da * da + db * db;
                if (mode == XI_DIFF) {
                    const float2 f = make_float2((float)da, (float)db);
                    dout[k] = f;
                    rout[k] = f;
                }
            }
            if (mode != XI_DIFF) out[k] = n;
        });
    };
    if (is_low(e)) emit(Low());
    else emit(NotLow());
    if (res) {
        const double s = cta_sum<T>(acc, red);
        if (threadIdx.x == 0) partial[(long long)slot * gridDim.x + blockIdx.x] = s;
    }
}

// x inverse of one sweep, field store and residual, polarization and x forward of the next, in
// place on the spectrum: the values and operations of k_fxx_inverse (XI_INPLACE_RES) followed by
// k_fxx_forward (XF_POLARIZE), without reading the field back (used where it is faster, see
// Solver::sweeps).
template <int M>
__global__ void __launch_bounds__(XShape<M>::T, min_ctas(XShape<M>::T, 896))
k_fxx_round(GridDesc g, unsigned mask, c64* spec, double* __restrict__ tau, double* __restrict__ partial) {
    using X = XShape<M>;
    using P = Plan<M>;
    using S = typename X::S;
    constexpr int N = X::N, RW = X::RW, TPP = X::TPP, T = X::T, J = M / P::R0;
    grid_begin();
    const int slot = blockIdx.y;
    if (!slot_active(g, mask, slot)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    c64* sm = reinterpret_cast<c64*>(smem_raw);
    __shared__ int key[2 * RW];
    __shared__ unsigned orm[5 * RW];   // inverse stages, forward stages, spectrum
    __shared__ double red[pow2_at_least(T)];
    const int r = threadIdx.x / TPP, t = threadIdx.x % TPP;
    for (int i = threadIdx.x; i < 5 * RW; i += T) {
        orm[i] = 0;
        if (i < 2 * RW) key[i] = kExpZero;
    }
    const long long row = (long long)slot * 3 * N * N + (long long)blockIdx.x * RW + r;   // slot, c, z, y
    c64* sp = spec + row * M;
    const uchar2* ph = reinterpret_cast<const uchar2*>(g.phase) + (long long)((int)(blockIdx.x * RW + r) % (N * N)) * M;
    __syncthreads();
    c64 v[P::I0][P::R0], o[P::IL][P::RL];
    int e;
    const bool bad = load_merge<M>(g, v, t, r, row, sp, key, e);
    transform<M, S>(v, o, t, r, sm, orm, RW, e, g.twf + N);
    e -= scale_bits(N);
    if (P::NS > 1) __syncthreads();   // the last stage has been read by every thread
    double2* out = reinterpret_cast<double2*>(tau) + row * M;
    const double cf[3] = {g.YN[0], g.YN[1], g.YN[2]};
    double acc = 0.0;
    int mk = kExpZero;
    // (loads first: one at a time between the stores they would each wait for memory, 3 to 5
    // times the kernel's time on grids beyond L2)
    double2 old[P::IL][P::RL];
    uchar2 pq[P::IL][P::RL];
    last_places<M>(t, [&](int k, int it, int q) {
        old[it][q] = out[k];
        pq[it][q] = ph[k];
    });
    const bool low = is_low(e);
    last_places<M>(t, [&](int k, int it, int q) {
        const c64 z = o[it][q];
        double2 n = low ? from_fixed<true>(swap_ri(z), e) : from_fixed(swap_ri(z), e);
        if (bad) n = make_double2(nan(""), nan(""));
        const double da = n.x - old[it][q].x, db = n.y - old[it][q].y;
        acc += da * da + db * db;
        out[k] = n;
        const uchar2 b = pq[it][q];
        n.x *= coef3(b.x, cf);
        n.y *= coef3(b.y, cf);
        mk = max(mk, max(key_of(n.x), key_of(n.y)));
        sm[S::at(k, r)] = mkc(__double_as_longlong(n.x), __double_as_longlong(n.y));
    });
    atomicMax(&key[RW + r], mk);
    __syncthreads();
    const int E = key[RW + r];
    e = E - first_bits(P::R0);
#pragma unroll
    for (int it = 0; it < P::I0; ++it)
        if (J % TPP == 0 || t + it * TPP < J) {
#pragma unroll
            for (int q = 0; q < P::R0; ++q) {
                const c64 d = sm[S::at(t + it * TPP + q * J, r)];
                v[it][q] = mkc(to_fixed(__longlong_as_double(d.x), e), to_fixed(__longlong_as_double(d.y), e));
            }
        }
    __syncthreads();
    transform<M, S>(v, o, t, r, sm, orm + 2 * RW, RW, e, g.twf + N);
    split_store<M>(g, o, t, r, row, sp, sm, orm + 4 * RW, E, e);
    const double s = cta_sum<T>(acc, red);
    if (threadIdx.x == 0) partial[(long long)slot * gridDim.x + blockIdx.x] = s;
}

// ---------------------------------------------------------------------------
// columns along y or z of one component: transform in place (y passes of a sweep; the z
// passes of a plain 3D transform, which read or write FP64 on their far side)
// ---------------------------------------------------------------------------
struct ColArgs {
    int inverse;
    const int* ein;
    int* eout;
};

template <int L>
struct ColShape {
    static constexpr int M = L / 2, NP = col_cols<L>(), TPP = Plan<L>::TPP, T = NP * TPP;
    using S = Slots<L, NP, false>;
    static constexpr size_t smem = sizeof(c64) * S::TOTAL;
};

// PLAIN: along z of each (component, ky) plane, from FP64 (inverse) or to FP64 (forward); else along y of
// each (component, z) plane, integers both ways (chosen at run time the FP64 side cost the y passes
// registers and code: a sweep of one gradient 29.1 us against 28.3 at 32^3, 1790 against 1712 at 256^3).
template <int L, bool PLAIN>
__global__ void __launch_bounds__(ColShape<L>::T, min_ctas(ColShape<L>::T, 1024))
k_fxx_col(GridDesc g, unsigned mask, const c64* src, c64* spec, ColArgs a) {
    using C = ColShape<L>;
    using P = Plan<L>;
    using S = typename C::S;
    constexpr int M = C::M, NP = C::NP, TPP = C::TPP, T = C::T, J = L / P::R0;
    grid_begin();
    const int slot = blockIdx.y;
    if (!slot_active(g, mask, slot)) return;
    const bool fp64_in = PLAIN && a.inverse, fp64_out = PLAIN && !a.inverse;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    c64* sm = reinterpret_cast<c64*>(smem_raw);
    __shared__ int key[NP];
    __shared__ unsigned orm[2 * NP];
    const int p = threadIdx.x % NP, t = threadIdx.x / NP;
    for (int i = threadIdx.x; i < 2 * NP; i += T) {
        orm[i] = 0;
        if (i < NP) key[i] = kExpZero;
    }
    const int kx = blockIdx.x % (M / NP) * NP + p;
    const int cw = blockIdx.x / (M / NP);                        // c L + z (y columns) or c L + ky (z columns)
    const long long plane = (long long)slot * 3 * L + cw;        // (slot, c, z) or (slot, c, ky)
    const long long comp = (long long)slot * 3 + cw / L;         // (slot, c)
    const long long first = PLAIN ? comp * L * L * M + (long long)(cw % L) * M + kx : plane * L * M + kx;
    const long long step = PLAIN ? (long long)L * M : M;
    const c64* in = src + first;   // the same buffer, or the FP64 spectrum of a plain inverse
    c64* base = spec + first;
    // exponent of element i: per (plane, y) for the y forward, per (component, i, kx) otherwise
    const int* ein = a.ein + (!PLAIN && !a.inverse ? plane * L : comp * L * M + kx);
    const int estep = !PLAIN && !a.inverse ? 1 : M;
    __syncthreads();
    c64 v[P::I0][P::R0];
    int mk = kExpZero;
#pragma unroll
    for (int it = 0; it < P::I0; ++it) {
        const int j = t + it * TPP;
        if (J % TPP == 0 || j < J) {
#pragma unroll
            for (int q = 0; q < P::R0; ++q) {
                const int i = j + q * J;
                v[it][q] = in[i * step];
                if (fp64_in)
                    mk = max(mk, max(key_of(__longlong_as_double(v[it][q].x)), key_of(__longlong_as_double(v[it][q].y))));
                else
                    mk = max(mk, ein[i * estep] + bits_of(mag(v[it][q])));
            }
        }
    }
    atomicMax(&key[p], mk);
    __syncthreads();
    const int E = key[p];
    int e = E - first_bits(P::R0);
#pragma unroll
    for (int it = 0; it < P::I0; ++it) {
        const int j = t + it * TPP;
        if (J % TPP == 0 || j < J) {
#pragma unroll
            for (int q = 0; q < P::R0; ++q) {
                c64 z = v[it][q];
                if (fp64_in) z = mkc(to_fixed(__longlong_as_double(z.x), e), to_fixed(__longlong_as_double(z.y), e));
                else z = shift(z, ein[(j + q * J) * estep] - e);
                v[it][q] = a.inverse ? swap_ri(z) : z;
            }
        }
    }
    c64 o[P::IL][P::RL];
    transform<L, S>(v, o, t, p, sm, orm, NP, e, g.twf);
    const bool bad = exp_is_nan(E);
    const double qn = bad ? nan("") : 0.0;
    auto emit = [&](auto f) {
        last_emit<L>(o, t, [&](int k, c64 z) { base[k * step] = f(a.inverse ? swap_ri(z) : z); });
    };
    auto bits = [&](double2 d) { return mkc(__double_as_longlong(d.x + qn), __double_as_longlong(d.y + qn)); };
    if (!fp64_out) emit([](c64 z) { return z; });
    else if (is_low(e)) emit([&](c64 z) { return bits(from_fixed<true>(z, e)); });
    else emit([&](c64 z) { return bits(from_fixed(z, e)); });
    if (t == 0 && !fp64_out) a.eout[plane * M + kx] = bad ? kExpNan : e;
}

// ---------------------------------------------------------------------------
// z pass of a sweep or an equilibrium test: forward along z for the three components, then
// the Green operator and the inverse (MODE Z_ITER, Z_ITER_NOB), or the divergence norm (Z_EQ)
// ---------------------------------------------------------------------------
template <int L>
struct ZShape {
    static constexpr int M = L / 2, NP = z_cols<L>(), P3 = 3 * NP, TPP = Plan<L>::TPP, T = P3 * TPP;
    using S = Slots<L, P3, false>;
    static constexpr size_t smem = sizeof(c64) * S::TOTAL;
};

// exponent b of the projector scale 4^b >= n2, b >= 1
__device__ __forceinline__ int proj_bits(int n2) { return max(1, (33 - __clz(n2 - 1)) >> 1); }

// (d . s) 2^-b rounded, |d| <= 2^b: exact products in two halves
__device__ __forceinline__ long long dir_dot(const long long* s, const int* d, int b) {
    const long long h = wide(hi_s(s[0]), d[0]) + (wide(hi_s(s[1]), d[1]) + wide(hi_s(s[2]), d[2]));
    const long long l = wide(lo_s(s[0]), d[0]) + (wide(lo_s(s[1]), d[1]) + (wide(lo_s(s[2]), d[2]) + ((1LL << b) >> 1)));
    return (long long)((unsigned long long)h << (32 - b)) + (l >> b);
}
// s <- ga s - 2^gs d (d . s) / |d|^2; G = 2^60 4^b / |d|^2
__device__ __forceinline__ void project(long long* s, const int* d, int b, long long G, int ga, int gs) {
    const long long D = dir_dot(s, d, b);
    const int dl = lo_s(D), dh = hi_s(D), gl = lo_s(G), gh = hi_s(G);
    const long long mid = wide(dh, gl) + (wide(dl, gh) + ((wide(dl, gl) >> 32) + (1LL << 27)));
    const long long T = (wide(dh, gh) << 4) + (mid >> 28);    // D 4^b / |d|^2
    const int tl = lo_s(T), th = hi_s(T), q = b - gs;
    const long long rnd = (1LL << q) >> 1;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const long long w = (long long)((unsigned long long)wide(th, d[c]) << (32 - q)) + ((wide(tl, d[c]) + rnd) >> q);
        s[c] = (ga ? s[c] : 0) - w;
    }
}

template <int L>
__global__ void __launch_bounds__(ZShape<L>::T, min_ctas(ZShape<L>::T, 1024))
k_fxx_z(GridDesc g, unsigned mask, int mode, c64* __restrict__ spec, double* __restrict__ partial) {
    using Z = ZShape<L>;
    using P = Plan<L>;
    using S = typename Z::S;
    constexpr int N = L, M = Z::M, NP = Z::NP, P3 = Z::P3, TPP = Z::TPP, T = Z::T, J = L / P::R0;
    grid_begin();
    const int slot = blockIdx.y;
    if (!slot_active(g, mask, slot)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    c64* sm = reinterpret_cast<c64*>(smem_raw);
    __shared__ int key[P3], ez[P3];
    __shared__ unsigned orm[5 * P3];   // forward stages, spectrum, inverse stages
    const int cp = threadIdx.x % P3, t = threadIdx.x / P3;
    for (int i = threadIdx.x; i < 5 * P3; i += T) {
        orm[i] = 0;
        if (i < P3) key[i] = kExpZero;
    }
    const int kx0 = blockIdx.x % (M / NP) * NP, ky = blockIdx.x / (M / NP);
    const long long comp = (long long)slot * 3 + cp / NP;        // (slot, c)
    c64* base = spec + comp * L * L * M + (long long)ky * M + kx0 + cp % NP;
    constexpr long long step = (long long)L * M;
    const int* ein = g.expB + comp * L * M + kx0 + cp % NP;      // exponent of plane z: ein[z M]
    __syncthreads();
    int e;
    c64 o[P::IL][P::RL];
    {
        c64 v[P::I0][P::R0];
        int mk = kExpZero;
#pragma unroll
        for (int it = 0; it < P::I0; ++it) {
            const int j = t + it * TPP;
            if (J % TPP == 0 || j < J) {
#pragma unroll
                for (int q = 0; q < P::R0; ++q) {
                    v[it][q] = base[(j + q * J) * step];
                    mk = max(mk, ein[(j + q * J) * M] + bits_of(mag(v[it][q])));
                }
            }
        }
        atomicMax(&key[cp], mk);
        __syncthreads();
        e = key[cp] - first_bits(P::R0);
#pragma unroll
        for (int it = 0; it < P::I0; ++it) {
            const int j = t + it * TPP;
            if (J % TPP == 0 || j < J) {
#pragma unroll
                for (int q = 0; q < P::R0; ++q) v[it][q] = shift(v[it][q], ein[(j + q * J) * M] - e);
            }
        }
        transform<L, S>(v, o, t, cp, sm, orm, P3, e, g.twf);
        if (P::NS > 1) __syncthreads();   // the last stage has been read by every thread
        unsigned m = 0;
        last_emit<L>(o, t, [&](int k, c64 z) {
            m |= mag(z);
            sm[S::at(k, cp)] = z;
        });
        atomicOr(&orm[2 * P3 + cp], m);
        if (t == 0) ez[cp] = e;
        __syncthreads();
    }
    // modes (kz, p): the three components share one scale per column (largest of the three)
    const int gs = g.gb == 2.0 ? 1 : 0, ga = g.ga != 0.0 ? 1 : 0;
    const bool addb = mode == Z_ITER;
    constexpr int BT = first_bits(P::R0) - 1;   // one bit for |s'_c| <= |s|
    double acc = 0.0;
    auto column_top = [&](int p) {   // exponent bound of the column's values
        int top = kExpZero;
#pragma unroll
        for (int c = 0; c < 3; ++c) top = max(top, ez[c * NP + p] + bits_of(orm[2 * P3 + c * NP + p]));
        if (kx0 + p == 0 && ky == 0 && addb)   // room for the mean added at DC
            for (int c = 0; c < 3; ++c)
                if (g.E[slot][c] != 0.0) top = max(top, ilogb(g.gc * g.E[slot][c]) + scale_bits(N) + 1);
        return kx0 + p == 0 ? top + 1 : top;
    };
    auto column_bad = [&](int p) {
        return exp_is_nan(key[p]) || exp_is_nan(key[NP + p]) || exp_is_nan(key[2 * NP + p]);
    };
    for (int q = threadIdx.x; q < L * NP; q += T) {
        const int p = q % NP, kz = q / NP, kx = kx0 + p;
        const int eg = column_top(p) - BT;
        c64 s[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) s[c] = shift(sm[S::at(kz, c * NP + p)], ez[c * NP + p] - eg);
        const int my = signed_mode(ky, N), mz = signed_mode(kz, N);
        const bool special = kx == 0 && (ky == 0 || ky == N / 2) && (kz == 0 || kz == N / 2);
        if (special) {   // four self-conjugate modes of the packed column, in FP64
            double2 f[3];
            for (int c = 0; c < 3; ++c) f[c] = from_fixed<true>(s[c], eg);
            if (mode == Z_EQ) {
                acc += eq_mode(kx, ky, kz, N, f[0], f[1], f[2]);
            } else {
                constexpr double up = (double)(1LL << scale_bits(N));   // gc E in the spectrum's scale
                const double cE[3] = {up * (g.gc * g.E[slot][0]), up * (g.gc * g.E[slot][1]), up * (g.gc * g.E[slot][2])};
                green_mode<double>(kx, ky, kz, N, 1.0, g.ga, g.gb, addb, cE, f[0], f[1], f[2]);
                for (int c = 0; c < 3; ++c) s[c] = mkc(to_fixed(f[c].x, eg), to_fixed(f[c].y, eg));
            }
        } else {
            int d[3];
            const int n2 = mode_dir(kx, my, mz, N, d);
            const int b = proj_bits(n2);
            long long re[3] = {s[0].x, s[1].x, s[2].x}, im[3] = {s[0].y, s[1].y, s[2].y};
            if (mode == Z_EQ) {
                // (squares of subnormals are zero)
                const double dr = from_fixed(dir_dot(re, d, b), eg + b), di = from_fixed(dir_dot(im, d, b), eg + b);
                acc += (kx == 0 ? 1.0 : 2.0) * (dr * dr + di * di);
            } else {
                const long long G = __ldg(&g.rcp[n2]);
                project(re, d, b, G, ga, gs);
                project(im, d, b, G, ga, gs);
#pragma unroll
                for (int c = 0; c < 3; ++c) s[c] = mkc(re[c], im[c]);
            }
        }
        if (mode != Z_EQ) {
#pragma unroll
            for (int c = 0; c < 3; ++c) sm[S::at(kz, c * NP + p)] = s[c];
        }
    }
    if (mode == Z_EQ) {
        if (threadIdx.x < NP && column_bad(threadIdx.x)) acc = nan("");
        __syncthreads();   // sm is free: the sum reuses it
        const double twopi_n = 6.283185307179586476925 / (double)N;
        const double s = cta_sum<T>(acc, reinterpret_cast<double*>(smem_raw)) * twopi_n * twopi_n /
                         ((double)g.N3 * (double)g.N3);
        if (threadIdx.x == 0) partial[(long long)slot * gridDim.x + blockIdx.x] = s;
        return;
    }
    __syncthreads();
    // inverse along z
    e = column_top(cp % NP) - BT;
    c64 v[P::I0][P::R0];
#pragma unroll
    for (int it = 0; it < P::I0; ++it) {
        const int j = t + it * TPP;
        if (J % TPP == 0 || j < J) {
#pragma unroll
            for (int q = 0; q < P::R0; ++q) v[it][q] = swap_ri(sm[S::at(j + q * J, cp)]);
        }
    }
    __syncthreads();
    transform<L, S>(v, o, t, cp, sm, orm + 3 * P3, P3, e, g.twf);
    last_emit<L>(o, t, [&](int k, c64 z) { base[k * step] = swap_ri(z); });
    if (t == 0) g.expA[(comp * L + ky) * M + kx0 + cp % NP] = column_bad(cp % NP) ? kExpNan : e;
}

// ---------------------------------------------------------------------------
// launchers of one length
// ---------------------------------------------------------------------------
template <class K, class... Args>
void launch(K kern, dim3 grid, int threads, size_t smem, cudaStream_t st, const GridDesc& g, Args... args) {
    if (smem > 32 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_kernel(small_grid(g, sizeof(double)), kern, grid, threads, smem, st, g, args...);
}

}  // namespace fx
}  // namespace hmg
