// FP64 transforms in block fixed point: 64-bit integers with one exponent per pencil.
//
// GB300 issues 2 FP64 operations per clock and SM, against 128 32-bit integer adds and 16
// 32x32+64 multiply-adds (IMAD.WIDE): measured, 0.63 T DFMA/s and 15.8 T 64-bit adds/s.  An
// FP64 pass is therefore bound by the FP64 pipe (97 % of a sweep; 9.7 ms per gradient at
// 256^3), and the same butterflies on 64-bit integers cost a tenth of that.
//
// Numbers.  A pencil (one 1D transform) holds complex integers v with a common exponent e,
// value v 2^e.  On load every pencil is scaled so that its largest component fills `first`
// bits (59 or 60, what the first radix can grow without overflow), so the quantum is at
// most 2^-58 of the pencil's largest value where FP64 arithmetic rounds each operation to
// 2^-53 of its own size.  Before each later radix the largest magnitude actually reached
// decides how far the values are shifted down (mostly not at all), so no bits are given up
// to worst-case growth.  Data twiddles carry 62 fractional bits.  A forward
// transform of N = 8 .. 72 errs by 3 to 7e-17 of its norm against long double, its rounding to
// FP64 included (test_gpu_fixed_accuracy.py bounds it by 1.1e-16 and 1.7e-16).
//
// Between passes the spectrum stays in integers, with the exponent of the pencil that wrote
// each value in a side array, so only the field side of the x passes converts to and from
// FP64.  Zeros and subnormals count as 2^-1021 when a pencil's scale is chosen, so subnormals keep
// their bits and zero pencils get a quantum below every double; pencils with an infinity or a NaN
// carry a very large exponent that marks everything computed from them as NaN.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "hmg_internal.h"

namespace hmg {
namespace fx {

struct __align__(16) c64 {
    long long x, y;
};

constexpr int kExpZero = -(1 << 20);   // below every key: where a maximum starts
constexpr int kExpNan = 1 << 20;       // exponent of a pencil that holds an infinity or a NaN
#define HMG_HD __host__ __device__ __forceinline__

HMG_HD bool exp_is_nan(int e) { return e > kExpNan / 2; }

HMG_HD c64 mkc(long long x, long long y) { return c64{x, y}; }
HMG_HD c64 operator+(c64 a, c64 b) { return c64{a.x + b.x, a.y + b.y}; }
HMG_HD c64 operator-(c64 a, c64 b) { return c64{a.x - b.x, a.y - b.y}; }
HMG_HD c64 mul_mi(c64 a) { return c64{a.y, -a.x}; }   // -i a
HMG_HD c64 swap_ri(c64 a) { return c64{a.y, a.x}; }   // conj(a) i: turns a forward DFT into an inverse one

// x = hi 2^32 + lo with lo signed
HMG_HD int lo_s(long long x) { return (int)(unsigned)(unsigned long long)x; }
HMG_HD int hi_s(long long x) {
    return (int)(unsigned)((unsigned long long)x >> 32) + (int)((unsigned)(unsigned long long)x >> 31);
}
HMG_HD long long wide(int a, int b) { return (long long)a * (long long)b; }

// x c for a constant |c| < 1/2 given as C = round(c 2^64); error below one unit
template <long long C>
HMG_HD long long mulq(long long x) {
    constexpr int cl = (int)(unsigned)(unsigned long long)C;
    constexpr int ch = (int)((C - (long long)cl) >> 32);
    const int xl = lo_s(x), xh = hi_s(x);
    const long long mid = wide(xh, cl) + (wide(xl, ch) + (1LL << 31));
    return wide(xh, ch) + (mid >> 32);
}
// constants as round(c 2^64); those above 1/2 as 1 - c
constexpr long long kQ1mR2 = 5402926248376769404LL;    // 1 - sqrt(1/2)
constexpr long long kQ1mH3 = 2471395088767036514LL;    // 1 - sqrt(3)/2
constexpr long long kQ1mC8 = 1404174782535421627LL;    // 1 - cos(pi/8)
constexpr long long kQS8 = 7059263338087549767LL;      // sin(pi/8)
constexpr long long kQ1mC40 = 4315718282406409839LL;   // 1 - cos(40 deg)
constexpr long long kQ1mS40 = 6589405544070453923LL;   // 1 - sin(40 deg)
constexpr long long kQC80 = 3203243492287910726LL;     // cos(80 deg)
constexpr long long kQ1mS80 = 280247492088382768LL;    // 1 - sin(80 deg)
constexpr long long kQ1mC20 = 1112474790118499113LL;   // 1 - cos(20 deg)
constexpr long long kQS20 = 6309158051982071155LL;     // sin(20 deg)

HMG_HD long long mul_r2(long long x) { return x - mulq<kQ1mR2>(x); }
HMG_HD long long mul_h3(long long x) { return x - mulq<kQ1mH3>(x); }
HMG_HD long long half(long long x) { return (x + 1) >> 1; }

// a (c - i s) with c = C or 1 - C (CM), s = S or 1 - S (SM)
template <long long C, bool CM, long long S, bool SM>
HMG_HD c64 rot(c64 a) {
    const long long cx = CM ? a.x - mulq<C>(a.x) : mulq<C>(a.x), cy = CM ? a.y - mulq<C>(a.y) : mulq<C>(a.y);
    const long long sx = SM ? a.x - mulq<S>(a.x) : mulq<S>(a.x), sy = SM ? a.y - mulq<S>(a.y) : mulq<S>(a.y);
    return c64{cx + sy, cy - sx};
}

// the same operations on FP32 pairs (hmg_gen32_kernels.cuh)
HMG_HD float2 mkc(float x, float y) { return make_float2(x, y); }
#ifdef __CUDA_ARCH__
HMG_HD float2 operator+(float2 a, float2 b) { return __fadd2_rn(a, b); }
HMG_HD float2 operator-(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
#else
HMG_HD float2 operator+(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
HMG_HD float2 operator-(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
#endif
HMG_HD float2 mul_mi(float2 a) { return make_float2(a.y, -a.x); }
HMG_HD float2 swap_ri(float2 a) { return make_float2(a.y, a.x); }
// Constants in two parts: rounded to FP32 they would scale every transform alike, and the error
// of the six passes of a sweep would add up with one sign (relative gain of a radix-9 DFT
// -1.6e-8 with rounded constants, below 1e-10 so; its rounding error 6.8e-8 and 6.3e-8).
HMG_HD float mul_r2(float x) {
    return fmaf(x, 0.70710678118654752f, x * (float)(0.70710678118654752 - 0.70710678118654752f));
}
HMG_HD float mul_h3(float x) {
    return fmaf(x, 0.86602540378443865f, x * (float)(0.86602540378443865 - 0.86602540378443865f));
}
HMG_HD float half(float x) { return 0.5f * x; }
template <long long C, bool CM, long long S, bool SM>
HMG_HD float2 rot(float2 a) {
    constexpr double u = 1.0 / 18446744073709551616.0;   // 2^-64
    constexpr double cd = CM ? 1.0 - (double)C * u : (double)C * u, sd = SM ? 1.0 - (double)S * u : (double)S * u;
    constexpr float c = (float)cd, cl = (float)(cd - c), s = (float)sd, sl = (float)(sd - s);
    return make_float2(fmaf(c, a.x, fmaf(s, a.y, fmaf(cl, a.x, sl * a.y))),
                       fmaf(c, a.y, -fmaf(s, a.x, fmaf(sl, a.x, -cl * a.y))));
}
template <class T>
HMG_HD T neg(T a) { return mkc(-a.x, -a.y); }
template <class T>
HMG_HD T rot8(T a) { return mkc(mul_r2(a.x + a.y), mul_r2(a.y - a.x)); }   // a exp(-i pi/4)

// a w / 4 for a table twiddle w = (r.h 2^-30 + r.l 2^-62) + i (...) : {r.h, r.l, i.h, i.l}
HMG_HD c64 cmul4(c64 a, int4 w) {
    const int xl = lo_s(a.x), xh = hi_s(a.x), yl = lo_s(a.y), yh = hi_s(a.y);
    const int nih = -w.z, nil = -w.w;
    const long long r = 1LL << 31;
    const long long mr = wide(yh, nil) + (wide(xh, w.y) + (wide(yl, nih) + (wide(xl, w.x) + r)));
    const long long mi = wide(yh, w.y) + (wide(xh, w.w) + (wide(yl, w.x) + (wide(xl, w.z) + r)));
    return c64{wide(yh, nih) + (wide(xh, w.x) + (mr >> 32)), wide(yh, w.x) + (wide(xh, w.z) + (mi >> 32))};
}
HMG_HD int4 conj_tw(int4 w) {
    w.z = -w.z;
    w.w = -w.w;
    return w;
}
HMG_HD c64 quarter(c64 a) { return c64{(a.x + 2) >> 2, (a.y + 2) >> 2}; }

// v / 2^s rounded, s in [0, 64]
HMG_HD long long shr_round(long long v, int s) { return s == 0 ? v : ((v >> (s - 1)) + 1) >> 1; }
// v 2^sh, rounded when sh < 0
HMG_HD long long shift(long long v, int sh) {
    if (sh >= 0) return (long long)((unsigned long long)v << (sh < 63 ? sh : 63));
    const int s = -sh < 64 ? -sh : 64;
    return ((v >> (s - 1)) + 1) >> 1;
}
HMG_HD c64 shift(c64 v, int sh) { return c64{shift(v.x, sh), shift(v.y, sh)}; }
HMG_HD c64 shr_round(c64 v, int s) { return c64{shr_round(v.x, s), shr_round(v.y, s)}; }

// the magnitude's high word (|v| <= 2^(32 + its bit length))
HMG_HD unsigned mag(long long v) {
    const int h = (int)(v >> 32);
    return (unsigned)(h ^ (h >> 31));
}
HMG_HD unsigned mag(c64 v) { return mag(v.x) | mag(v.y); }
HMG_HD int clz32(unsigned v) {
#ifdef __CUDA_ARCH__
    return __clz((int)v);
#else
    return v ? __builtin_clz(v) : 32;
#endif
}
HMG_HD int clz64(unsigned long long v) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}
HMG_HD int bits_of(unsigned m) { return 64 - clz32(m); }   // of the full 64-bit magnitude
HMG_HD unsigned long long dbits(double d) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(d);
#else
    unsigned long long u;
    __builtin_memcpy(&u, &d, 8);
    return u;
#endif
}
HMG_HD double bitsd(unsigned long long u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double d;
    __builtin_memcpy(&d, &u, 8);
    return d;
#endif
}
// E with |d| < 2^E, the smallest for normal numbers; zeros and subnormals share -1021
HMG_HD int key_of(double d) {
    const unsigned long long u = dbits(d);
    const int ex = (int)((u >> 52) & 0x7ff);
    return ex == 2047 ? kExpNan : (ex ? ex : 1) - 1022;
}
// round(d 2^-e) for |d| < 2^(e + 61)
HMG_HD long long to_fixed(double d, int e) {
    const unsigned long long u = dbits(d);
    const int ex = (int)((u >> 52) & 0x7ff);
    // 1.f (0.f) at bit 62
    const unsigned long long m = ((u << 10) & 0x3ffffffffffffc00ull) | ((unsigned long long)(ex ? 1u << 30 : 0u) << 32);
    int r = e + 1084 - (ex ? ex : 1);          // one less than the right shift
    r = r < 0 ? 0 : (r > 63 ? 63 : r);
    const long long v = (long long)(((m >> r) + 1) >> 1);
    const long long s = (long long)u >> 63;
    return (v ^ s) - s;
}
// Values of a pencil with quantum 2^e may be subnormal where is_low(e).  LOW: with subnormals, else they
// count as zero.  (A template parameter and a branch per pencil: tested per value they cost
// every pass, a sweep at 256^3 10 %.)
HMG_HD bool is_low(int e) { return e < -1022; }
// v 2^e as a double, rounded to nearest
template <bool LOW = false>
HMG_HD double from_fixed(long long v, int e) {
    const long long s = v >> 63;
    const unsigned long long a = (unsigned long long)((v ^ s) - s);
    const int lz = clz64(a);
    const unsigned long long n = a << (lz & 63);
    const int ex = e + 1085 - lz;              // biased exponent, less one (the leading bit adds it)
    unsigned long long b = (n >> 11) + ((n >> 10) & 1) + ((unsigned long long)(unsigned)ex << 52);
    if (ex >= 2046) b = 0x7ff0000000000000ull;
    if (ex < 0 || a == 0) b = LOW ? (unsigned long long)shift((long long)a, e + 1074) : 0;
    return bitsd(b | ((unsigned long long)s & 0x8000000000000000ull));
}
template <bool LOW = false>
HMG_HD double2 from_fixed(c64 v, int e) { return make_double2(from_fixed<LOW>(v.x, e), from_fixed<LOW>(v.y, e)); }
using Low = std::true_type;
using NotLow = std::false_type;

// ---------------------------------------------------------------------------
// forward DFTs of small length in registers, natural order in and out
// ---------------------------------------------------------------------------
template <int R> struct Dft;
template <> struct Dft<2> {
    template <class T> HMG_HD static void run(T* v) {
        const T a = v[0];
        v[0] = a + v[1];
        v[1] = a - v[1];
    }
};
template <> struct Dft<3> {
    template <class T> HMG_HD static void run(T* v) {
        const T t = v[1] + v[2], u = v[1] - v[2];
        const T m = mkc(v[0].x - half(t.x), v[0].y - half(t.y));
        const T h = mkc(mul_h3(u.y), -mul_h3(u.x));   // -i sqrt(3)/2 u
        v[0] = v[0] + t;
        v[1] = m + h;
        v[2] = m - h;
    }
};
template <> struct Dft<4> {
    template <class T> HMG_HD static void run(T* v) {
        const T a = v[0] + v[2], b = v[0] - v[2], c = v[1] + v[3], d = mul_mi(v[1] - v[3]);
        v[0] = a + c;
        v[1] = b + d;
        v[2] = a - c;
        v[3] = b - d;
    }
};
template <> struct Dft<8> {
    template <class T> HMG_HD static void run(T* v) {
        T a[4], b[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            a[r] = v[r] + v[r + 4];
            b[r] = v[r] - v[r + 4];
        }
        b[1] = rot8(b[1]);
        b[2] = mul_mi(b[2]);
        b[3] = mul_mi(rot8(b[3]));
        Dft<4>::run(a);
        Dft<4>::run(b);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            v[2 * r] = a[r];
            v[2 * r + 1] = b[r];
        }
    }
};
template <> struct Dft<9> {
    template <class T> HMG_HD static void run(T* v) {
        T s[3][3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
#pragma unroll
            for (int a = 0; a < 3; ++a) s[b][a] = v[3 * a + b];
            Dft<3>::run(s[b]);
        }
        s[1][1] = rot<kQ1mC40, true, kQ1mS40, true>(s[1][1]);
        s[1][2] = rot<kQC80, false, kQ1mS80, true>(s[1][2]);
        s[2][1] = rot<kQC80, false, kQ1mS80, true>(s[2][1]);
        // exp(-i 160 deg) = -i exp(-i 70 deg), cos 70 = sin 20, sin 70 = cos 20
        s[2][2] = mul_mi(rot<kQS20, false, kQ1mC20, true>(s[2][2]));
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            T t[3] = {s[0][k], s[1][k], s[2][k]};
            Dft<3>::run(t);
            v[k] = t[0];
            v[k + 3] = t[1];
            v[k + 6] = t[2];
        }
    }
};
template <> struct Dft<16> {
    template <class T> HMG_HD static void run(T* v) {
        T s[4][4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
#pragma unroll
            for (int a = 0; a < 4; ++a) s[b][a] = v[4 * a + b];
            Dft<4>::run(s[b]);
        }
        s[1][1] = rot<kQ1mC8, true, kQS8, false>(s[1][1]);
        s[1][2] = rot8(s[1][2]);
        s[1][3] = rot<kQS8, false, kQ1mC8, true>(s[1][3]);
        s[2][1] = rot8(s[2][1]);
        s[2][2] = mul_mi(s[2][2]);
        s[2][3] = mul_mi(rot8(s[2][3]));
        s[3][1] = rot<kQS8, false, kQ1mC8, true>(s[3][1]);
        s[3][2] = mul_mi(rot8(s[3][2]));
        s[3][3] = neg(rot<kQ1mC8, true, kQS8, false>(s[3][3]));   // exp(-i 9 pi/8)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            T t[4] = {s[0][k], s[1][k], s[2][k], s[3][k]};
            Dft<4>::run(t);
#pragma unroll
            for (int q = 0; q < 4; ++q) v[k + 4 * q] = t[q];
        }
    }
};
// R = A B with coprime factors: index maps without twiddles (Good 1958).  Input n = B a + A b
// mod R, output k = U a' + V b' mod R with U = 1 mod A, 0 mod B and V = 0 mod A, 1 mod B.
template <int A, int B>
struct CoprimeDft {
    static constexpr int R = A * B;
    HMG_HD static constexpr int unit(int one, int zero) {
        int u = zero;
        while (u % one != 1) u += zero;
        return u;
    }
    template <class T> HMG_HD static void run(T* v) {
        constexpr int U = unit(A, B), V = unit(B, A);
        T s[B][A];
#pragma unroll
        for (int b = 0; b < B; ++b) {
#pragma unroll
            for (int a = 0; a < A; ++a) s[b][a] = v[(B * a + A * b) % R];
            Dft<A>::run(s[b]);
        }
#pragma unroll
        for (int a = 0; a < A; ++a) {
            T t[B];
#pragma unroll
            for (int b = 0; b < B; ++b) t[b] = s[b][a];
            Dft<B>::run(t);
#pragma unroll
            for (int b = 0; b < B; ++b) v[(U * a + V * b) % R] = t[b];
        }
    }
};
template <> struct Dft<6> : CoprimeDft<2, 3> {};
template <> struct Dft<12> : CoprimeDft<4, 3> {};
template <> struct Dft<18> : CoprimeDft<2, 9> {};
template <> struct Dft<24> : CoprimeDft<8, 3> {};

// Component bits a radix may start from: R 2^(b + 1/2) < 2^63 without twiddles (`first`),
// R 2^(b + 1/2) / 4 < 2^63 and b <= 62 behind the /4 of the twiddle product (`later`).
constexpr int first_bits(int R) { return R >= 6 ? 59 : R >= 3 ? 60 : 61; }   // (R <= 9 in every plan)
constexpr int later_bits(int R) { return R >= 6 ? 61 : 62; }

// Radices of a length (first stage first, 1 = no stage) and threads per pencil: every
// thread takes whole radix butterflies, one to three per stage.  Three stages of at most 8
// or 9 values instead of two of up to 16: 64 registers instead of 128 and so twice the
// warps, which hide the loads and the integer latency better than the third exchange costs
// (one sweep of one gradient, kernels alone: 256^3 2.20 -> 1.88 ms, 192^3 1.56 -> 0.92 ms,
// 512^3 23.4 -> 16.5 ms).
template <int R0_, int R1_, int R2_, int T_>
struct PlanOf {
    static constexpr int R0 = R0_, R1 = R1_, R2 = R2_, TPP = T_;
    static constexpr int NS = R2_ > 1 ? 3 : R1_ > 1 ? 2 : 1;
    static constexpr int L = R0_ * R1_ * R2_;
    static constexpr int I0 = (L / R0_ + T_ - 1) / T_, I1 = (L / R1_ + T_ - 1) / T_, I2 = (L / R2_ + T_ - 1) / T_;
    // the last stage: radix, butterflies per thread, product of the stages before it
    static constexpr int RL = NS == 3 ? R2_ : NS == 2 ? R1_ : R0_;
    static constexpr int IL = NS == 3 ? I2 : NS == 2 ? I1 : I0;
    static constexpr int NL = L / RL;
};
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
template <> struct Plan<32> : PlanOf<4, 4, 2, 8> {};
template <> struct Plan<36> : PlanOf<6, 6, 1, 6> {};
template <> struct Plan<48> : PlanOf<4, 4, 3, 12> {};
template <> struct Plan<54> : PlanOf<9, 6, 1, 9> {};
template <> struct Plan<64> : PlanOf<8, 8, 1, 8> {};
template <> struct Plan<72> : PlanOf<9, 8, 1, 9> {};
template <> struct Plan<81> : PlanOf<9, 9, 1, 9> {};
template <> struct Plan<96> : PlanOf<8, 4, 3, 12> {};
template <> struct Plan<108> : PlanOf<6, 6, 3, 18> {};
template <> struct Plan<128> : PlanOf<8, 4, 4, 16> {};
template <> struct Plan<144> : PlanOf<6, 6, 4, 24> {};
template <> struct Plan<162> : PlanOf<9, 6, 3, 27> {};
template <> struct Plan<192> : PlanOf<8, 6, 4, 24> {};
template <> struct Plan<216> : PlanOf<6, 6, 6, 36> {};
template <> struct Plan<243> : PlanOf<9, 9, 3, 27> {};
template <> struct Plan<256> : PlanOf<8, 8, 4, 32> {};
template <> struct Plan<288> : PlanOf<6, 6, 8, 48> {};
template <> struct Plan<324> : PlanOf<9, 6, 6, 54> {};
template <> struct Plan<384> : PlanOf<8, 8, 6, 64> {};
template <> struct Plan<432> : PlanOf<9, 8, 6, 72> {};
template <> struct Plan<486> : PlanOf<9, 9, 6, 81> {};
template <> struct Plan<512> : PlanOf<8, 8, 8, 64> {};

// Shared-memory slots of a pencil.  Columns: NPEN pencils interleaved (index-major), so
// neighbouring threads touch neighbouring 16-byte slots.  Rows: one pencil after another,
// padded by one slot per R0 values where R0 is even, so that the first stage's stores (a
// stride of R0 slots between threads) fall on distinct banks.
template <int L, int NPEN, bool ROW>
struct Slots {
    static constexpr int PAD = (ROW && Plan<L>::R0 % 2 == 0) ? Plan<L>::R0 : 0;
    static constexpr int LEN = PAD ? L + L / PAD : L;
    static constexpr int TOTAL = LEN * NPEN;
    HMG_HD static int at(int i, int pen) {
        if constexpr (ROW) return pen * LEN + (PAD ? i + i / (PAD ? PAD : 1) : i);
        else return i * NPEN + pen;
    }
};

#ifdef __CUDACC__
// One later stage of radix R behind stages of product NSP: read, shift, twiddle, DFT.
template <int L, int R, int NSP, int IT, class S>
__device__ __forceinline__ void stage_read(c64 (&v)[IT][R], int t, int pen, const c64* sm, int sh,
                                           const int4* __restrict__ tw) {
    constexpr int TPP = Plan<L>::TPP, J = L / R, TS = L / (NSP * R);
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int j = t + it * TPP;
        if (J % TPP == 0 || j < J) {
            const int k = j % NSP;
#pragma unroll
            for (int r = 0; r < R; ++r) v[it][r] = sm[S::at(j + r * J, pen)];
            if (sh) {
#pragma unroll
                for (int r = 0; r < R; ++r) v[it][r] = shr_round(v[it][r], sh);
            }
            v[it][0] = quarter(v[it][0]);
#pragma unroll
            for (int r = 1; r < R; ++r) v[it][r] = cmul4(v[it][r], __ldg(&tw[k * r * TS]));
            Dft<R>::run(v[it]);
        }
    }
}
template <int L, int R, int NSP, int IT, class F>
__device__ __forceinline__ void stage_emit(const c64 (&v)[IT][R], int t, F f) {
    constexpr int TPP = Plan<L>::TPP, J = L / R;
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int j = t + it * TPP;
        if (J % TPP == 0 || j < J) {
            const int base = (j / NSP) * NSP * R + j % NSP;
#pragma unroll
            for (int r = 0; r < R; ++r) f(base + r * NSP, v[it][r]);
        }
    }
}

// Forward transform of one pencil by its TPP threads.  v: the first stage's inputs,
// v[it][r] = x[t + it TPP + r L / R0], in at most first_bits(R0) bits, exponent e; the outputs
// stay in the last stage's registers `o` (exponent e on return): last_emit<L> names their
// indices.  `or_max`: NS - 1 zeroed words per pencil (stride npen).  The buffer must be free
// on entry and may still be read by other threads on return.
template <int L, class S>
__device__ __forceinline__ void transform(c64 (&v)[Plan<L>::I0][Plan<L>::R0], c64 (&o)[Plan<L>::IL][Plan<L>::RL], int t,
                                          int pen, c64* sm, unsigned* or_max, int npen, int& e,
                                          const int4* __restrict__ tw) {
    using P = Plan<L>;
#pragma unroll
    for (int it = 0; it < P::I0; ++it)
        if ((L / P::R0) % P::TPP == 0 || t + it * P::TPP < L / P::R0) Dft<P::R0>::run(v[it]);
    if constexpr (P::NS == 1) {
#pragma unroll
        for (int it = 0; it < P::I0; ++it)
#pragma unroll
            for (int r = 0; r < P::R0; ++r) o[it][r] = v[it][r];
    } else {
        unsigned m = 0;
        stage_emit<L, P::R0, 1, P::I0>(v, t, [&](int k, c64 z) {
            m |= mag(z);
            sm[S::at(k, pen)] = z;
        });
        atomicOr(&or_max[pen], m);
        __syncthreads();
        int sh = max(0, bits_of(or_max[pen]) - later_bits(P::R1));
        if constexpr (P::NS == 2) {
            stage_read<L, P::R1, P::R0, P::I1, S>(o, t, pen, sm, sh, tw);
            e += 2 + sh;
        } else {
            c64 u[P::I1][P::R1];
            stage_read<L, P::R1, P::R0, P::I1, S>(u, t, pen, sm, sh, tw);
            e += 2 + sh;
            __syncthreads();   // every thread has read the previous stage
            m = 0;
            stage_emit<L, P::R1, P::R0, P::I1>(u, t, [&](int k, c64 z) {
                m |= mag(z);
                sm[S::at(k, pen)] = z;
            });
            atomicOr(&or_max[npen + pen], m);
            __syncthreads();
            sh = max(0, bits_of(or_max[npen + pen]) - later_bits(P::R2));
            stage_read<L, P::R2, P::R0 * P::R1, P::I2, S>(o, t, pen, sm, sh, tw);
            e += 2 + sh;
        }
    }
}
// f(index, butterfly, value) over the places of the last stage's registers
template <int L, class F>
__device__ __forceinline__ void last_places(int t, F f) {
    using P = Plan<L>;
    constexpr int J = L / P::RL;
#pragma unroll
    for (int it = 0; it < P::IL; ++it) {
        const int j = t + it * P::TPP;
        if (J % P::TPP == 0 || j < J) {
            const int base = (j / P::NL) * P::NL * P::RL + j % P::NL;
#pragma unroll
            for (int r = 0; r < P::RL; ++r) f(base + r * P::NL, it, r);
        }
    }
}
template <int L, class F>
__device__ __forceinline__ void last_emit(const c64 (&o)[Plan<L>::IL][Plan<L>::RL], int t, F f) {
    stage_emit<L, Plan<L>::RL, Plan<L>::NL, Plan<L>::IL>(o, t, f);
}
#endif  // __CUDACC__

}  // namespace fx
}  // namespace hmg
