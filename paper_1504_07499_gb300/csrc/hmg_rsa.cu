// Seeded sphere placement on the GPU (§2: up to 100 identical, non-overlapping spheres in
// the periodic unit cube, produced by random sequential adsorption), and the RVE
// pipeline placement -> voxelization.
//
// Random numbers: SplitMix64 (Steele, Lea & Flood, OOPSLA 2014) as a counter-based
// stream: output i (i >= 1) of stream s of a seed is mix(base + i * 0x9E3779B97F4A7C15)
// with base = seed + s * 0xD1B54A32D192ED03 (mod 2^64); a uniform double is the top 53
// bits times 2^-53.  Candidate j of a placement run takes outputs 3j+1, 3j+2, 3j+3.
//
// Placement (the same steps as the library's seeded host generator):
//   1. RSA at the target radius r (stream 0): candidates are accepted in draw order when
//      their periodic minimum-image distance to every accepted centre exceeds 2r (squared
//      distances against (2r)^2); candidates are drawn in blocks of 8192 until n spheres
//      are placed or a block ends at or past the candidate cap.
//   2. Above the RSA jamming limit (step 1 fails): RSA at 0.85 r (stream 2), then
//      Monte-Carlo displacement sweeps (stream 1) that let the radius grow: each sweep
//      sets the working radius to min(r, half the smallest pair distance) and stops once
//      it reaches r with every pair farther apart than 2r; otherwise every sphere in turn
//      tries a move by step (2u - 1) per axis (step = max(r/4, 1e-3), coordinates wrapped
//      into [0, 1) as fmod(x, 1) + 1 for negative remainders), kept when it stays farther
//      than twice the working radius from all others; each sweep draws 4 uniforms per
//      sphere (the fourth is unused).
// Squared distances are (dx^2 + dy^2) + dz^2 with d = min(|a - b|, 1 - |a - b|), every
// operation rounded on its own, so the sphere lists equal the host generator's bit for
// bit.  Every loop is bounded (candidate cap, sweep cap); failure is a status, not a hang.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "../../include/hmg.h"
#include "hmg_runtime.h"

namespace hmg {
namespace rsa {

constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;
constexpr uint64_t kStream = 0xD1B54A32D192ED03ull;
constexpr int kBlock = 8192;       // candidates per draw block
constexpr int kThreads = 1024;     // candidates examined per CTA round
constexpr int kMaxSpheres = 1024;  // shared-memory capacity of the kernels

__device__ __forceinline__ uint64_t mix(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__device__ __forceinline__ double uniform(uint64_t base, uint64_t counter) {
    return (double)(mix(base + counter * kGamma) >> 11) * 0x1.0p-53;
}
__device__ __forceinline__ double axis_d(double a, double b) {
    const double d = fabs(__dsub_rn(a, b));
    return fmin(d, __dsub_rn(1.0, d));
}
__device__ __forceinline__ double min_image_sq(double ax, double ay, double az, double bx, double by, double bz) {
    const double dx = axis_d(ax, bx), dy = axis_d(ay, by), dz = axis_d(az, bz);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// FP32 view of a centre and the squared minimum-image distance it gives.  Each coordinate in
// [0, 1] is off by at most 2^-25, a distance by 2^-23, the squared sum by less than 5e-7; so a
// comparison with a limit is decided by FP32 unless the two lie within kMargin, where the
// FP64 value decides.  (GB300 issues 64 times as many FP32 as FP64 operations.)
constexpr float kMargin = 1e-6f;
__device__ __forceinline__ float4 narrow(double x, double y, double z) {
    return make_float4((float)x, (float)y, (float)z, 0.f);
}
__device__ __forceinline__ float near_sq(float4 a, float4 b) {
    float dx = fabsf(a.x - b.x), dy = fabsf(a.y - b.y), dz = fabsf(a.z - b.z);
    dx = fminf(dx, 1.f - dx);
    dy = fminf(dy, 1.f - dy);
    dz = fminf(dz, 1.f - dz);
    return dx * dx + dy * dy + dz * dz;
}
// min_image_sq(a, b) > lim; p, q: the centres' FP64 coordinates
__device__ __forceinline__ bool clear_of(float4 a, float4 b, const double* p, const double* q, float limf, double lim) {
    const float f = near_sq(a, b);
    if (fabsf(f - limf) > kMargin) return f > limf;
    return min_image_sq(p[0], p[1], p[2], q[0], q[1], q[2]) > lim;
}

// Sequential RSA in one CTA.  Each round examines kThreads candidates in parallel against the
// accepted centres, then accepts them in draw order: the first candidate still clear is
// accepted and the later ones are re-examined against it only.  The candidates are items
// begin .. limit - 1, or, with a list, the candidates list[0 .. limit - 1], which the filter has
// found clear of the first `known` centres.
// out: 3 n doubles, the first state[0] centres placed before; state[0] = spheres placed.
__global__ void __launch_bounds__(kThreads) k_rsa(uint64_t base, int n, double lim, long long begin, long long limit,
                                                  const int* __restrict__ list, long long list_base,
                                                  double* __restrict__ out, long long* __restrict__ state) {
    __shared__ double acc[3 * kMaxSpheres];
    __shared__ float4 accf[kMaxSpheres];
    __shared__ int wfirst[kThreads / 32];
    __shared__ int s_first, s_count;
    const int t = threadIdx.x;
    const float limf = (float)lim;
    const int known = (int)state[0];
    if (list) limit = min(limit, state[2]);
    for (int i = t; i < 3 * known; i += kThreads) acc[i] = out[i];
    if (t == 0) s_count = known;
    __syncthreads();
    for (int i = t; i < known; i += kThreads) accf[i] = narrow(acc[3 * i], acc[3 * i + 1], acc[3 * i + 2]);
    __syncthreads();
    for (long long j0 = begin; j0 < limit && s_count < n; j0 += kThreads) {
        const bool valid = j0 + t < limit;
        const long long j = !valid ? 0 : list ? list_base + list[j0 + t] : j0 + t;
        double c[3] = {0.0, 0.0, 0.0};
        bool ok = valid;
        float4 cf = make_float4(0.f, 0.f, 0.f, 0.f);
        if (valid) {
#pragma unroll
            for (int a = 0; a < 3; ++a) c[a] = uniform(base, 3 * (uint64_t)j + 1 + a);
            cf = narrow(c[0], c[1], c[2]);
            for (int a = list ? known : 0; a < s_count && ok; ++a) ok = clear_of(cf, accf[a], c, acc + 3 * a, limf, lim);
        }
        int start = 0;
        bool round_done = false;
        while (!round_done) {   // at most kThreads acceptances per round
            const unsigned bal = __ballot_sync(0xffffffffu, ok && t >= start);
            if ((t & 31) == 0) wfirst[t >> 5] = bal ? (t & ~31) + __ffs(bal) - 1 : kThreads;
            __syncthreads();
            if (t < 32) {
                const int f = __reduce_min_sync(0xffffffffu, wfirst[t]);
                if (t == 0) s_first = f;
            }
            __syncthreads();
            const int f = s_first;
            if (f >= kThreads) {
                round_done = true;
            } else {
                if (t == f) {
                    const int a = s_count;
                    for (int i = 0; i < 3; ++i) acc[3 * a + i] = c[i];
                    accf[a] = cf;
                    s_count = a + 1;
                }
                __syncthreads();
                const int a = s_count - 1;
                if (ok && t > f) ok = clear_of(cf, accf[a], c, acc + 3 * a, limf, lim);
                if (t == f) ok = false;
                start = f + 1;
                if (s_count >= n) {
                    round_done = true;
                }
            }
            __syncthreads();
        }
    }
    for (int i = t; i < 3 * s_count; i += kThreads) out[i] = acc[i];
    if (t == 0) state[0] = s_count;
}

// After the first block most spheres are placed and nearly every candidate is rejected by one of
// them, so the rest of the draws goes through the whole GPU: kChunk candidates are tested
// against the centres placed so far (one bit each), the survivors are listed in draw order,
// and the sequential kernel examines only these against each other.  100 spheres at 40 %, which
// RSA cannot place in 400 000 candidates: one CTA took 3.9 ms over them; with this and the
// growth kernel's settled trials the whole call went from 12.4 to 6.1 ms.
constexpr int kChunk = 1 << 17;      // candidates per filter launch
constexpr int kSurvivors = 4096;     // listed at most; the next chunk starts behind the last one listed
__global__ void __launch_bounds__(256) k_rsa_filter(uint64_t base, double lim, long long begin, int count,
                                                    const double* __restrict__ centres,
                                                    const long long* __restrict__ state, unsigned* __restrict__ bits) {
    __shared__ float4 accf[kMaxSpheres];
    const int placed = (int)state[0];
    const float limf = (float)lim;
    for (int i = threadIdx.x; i < placed; i += 256) accf[i] = narrow(centres[3 * i], centres[3 * i + 1], centres[3 * i + 2]);
    __syncthreads();
    const int i = blockIdx.x * 256 + threadIdx.x;
    bool ok = i < count;
    if (ok) {
        double c[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) c[a] = uniform(base, 3 * (uint64_t)(begin + i) + 1 + a);
        const float4 cf = narrow(c[0], c[1], c[2]);
        for (int a = 0; a < placed && ok; ++a) ok = clear_of(cf, accf[a], c, centres + 3 * a, limf, lim);
    }
    const unsigned w = __ballot_sync(0xffffffffu, ok);
    if ((threadIdx.x & 31) == 0 && i < count) bits[i >> 5] = w;
}
// Survivors of `count` candidates in order: list (offsets from the chunk's first candidate),
// state[2] = how many are listed, state[3] = candidates of the chunk that are settled by them.
__global__ void __launch_bounds__(kThreads) k_rsa_list(const unsigned* __restrict__ bits, int count, int* __restrict__ list,
                                                       long long* __restrict__ state) {
    __shared__ int part[kThreads];
    const int words = (count + 31) / 32, t = threadIdx.x;
    const int per = (words + kThreads - 1) / kThreads, w0 = min(t * per, words), w1 = min(w0 + per, words);
    int c = 0;
    for (int w = w0; w < w1; ++w) c += __popc(bits[w]);
    part[t] = c;
    __syncthreads();
    for (int o = 1; o < kThreads; o <<= 1) {   // inclusive prefix sum
        const int add = t >= o ? part[t - o] : 0;
        __syncthreads();
        part[t] += add;
        __syncthreads();
    }
    int at = part[t] - c;
    const int total = part[kThreads - 1];
    for (int w = w0; w < w1 && at < kSurvivors; ++w)
        for (unsigned m = bits[w]; m && at < kSurvivors; m &= m - 1, ++at) {
            const int i = 32 * w + __ffs(m) - 1;
            list[at] = i;
            if (at == kSurvivors - 1) state[3] = i + 1;
        }
    if (t == 0) {
        state[2] = min(total, kSurvivors);
        if (total < kSurvivors) state[3] = count;
    }
}

// x in (-1, 2) wrapped into [0, 1): the exact remainder fmod(x, 1), plus 1 when it is negative
// (a zero remainder is +0)
__device__ __forceinline__ double wrap1(double x) {
    const double m = x >= 1.0 ? __dsub_rn(x, 1.0) : x;   // exact
    return m < 0.0 ? __dadd_rn(m, 1.0) : (m > 0.0 ? m : 0.0);
}

// Growth sweeps in one CTA.  A sweep is sequential by definition: sphere i's trial is tested
// against the moved spheres before it and the unmoved ones after it.  But every trial is
// known at the start of the sweep (a sphere moves once per sweep and its draw depends on its
// own position only), so whether trial i is clear of sphere k before (A) and after (B) k's
// own move is tabulated in parallel as bit rows.  That settles most trials; one warp walks the
// others in order with bit operations: trial i is taken when every k is clear, B where k < i
// has moved, A elsewhere.  Rows come in blocks of kRows spheres so that the tables of 1024
// spheres fit; B is needed only within a block (earlier blocks have settled before it).  Bound
// by the barriers and latency of one CTA.  100 spheres at 40 % through the C ABI, placement and
// 128^3 grid: 219 ms with FP64 distances and two barriers per sphere, 12.4 ms with the bit
// tables, 6.1 ms with settled trials and the filtered candidates above.
// c: 3 n doubles in/out; state[0] = 1 on success, state[1] = sweeps run.
constexpr int kRows = 128;
struct GrowSmem {
    double p[3 * kMaxSpheres];        // centres
    double tr[3 * kMaxSpheres];       // trials of the sweep
    float4 pf[kMaxSpheres], tf[kMaxSpheres];
    unsigned A[kRows][kMaxSpheres / 32];
    unsigned B[kRows][kMaxSpheres / 32];
    unsigned acc[kRows / 32];         // taken trials of the block
    unsigned open[kRows / 32];        // trials that depend on the order
    float wminf[kThreads / 32];
    double wmin[kThreads / 32];
    double lim;
    float dminf;
    int done;
};

__global__ void __launch_bounds__(kThreads) k_grow(uint64_t base, int n, double r_target, double lim_target,
                                                   int max_sweeps, double* __restrict__ c,
                                                   long long* __restrict__ state) {
    extern __shared__ __align__(16) unsigned char grow_raw[];
    GrowSmem& s = *reinterpret_cast<GrowSmem*>(grow_raw);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    constexpr int kWarps = kThreads / 32;
    for (int i = t; i < 3 * n; i += kThreads) s.p[i] = c[i];
    if (t == 0) s.done = 0;
    __syncthreads();
    for (int i = t; i < n; i += kThreads) s.pf[i] = narrow(s.p[3 * i], s.p[3 * i + 1], s.p[3 * i + 2]);
    const double step = fmax(__dmul_rn(0.25, r_target), 1e-3);
    const int words = (n + 31) / 32;
    int sweep = 0;
    __syncthreads();
    for (; sweep < max_sweeps; ++sweep) {
        // smallest squared pair distance: FP32 over all pairs, FP64 for those within the margins
        // of the smallest (a minimum does not depend on the order)
        float mf = INFINITY;
        for (int i = warp; i < n; i += kWarps) {
            const float4 a = s.pf[i];
            for (int k = lane; k < i; k += 32) mf = fminf(mf, near_sq(a, s.pf[k]));
        }
        const float own = mf;
        for (int o = 16; o > 0; o >>= 1) mf = fminf(mf, __shfl_xor_sync(0xffffffffu, mf, o));
        if (lane == 0) s.wminf[warp] = mf;
        __syncthreads();
        mf = s.wminf[lane];
        for (int o = 16; o > 0; o >>= 1) mf = fminf(mf, __shfl_xor_sync(0xffffffffu, mf, o));
        double m = INFINITY;
        if (own <= mf + 2.f * kMargin)   // this thread saw a pair near the minimum: scan its pairs again
            for (int i = warp; i < n; i += kWarps) {
                const float4 a = s.pf[i];
                for (int k = lane; k < i; k += 32)
                    if (near_sq(a, s.pf[k]) <= mf + 2.f * kMargin)
                        m = fmin(m, min_image_sq(s.p[3 * i], s.p[3 * i + 1], s.p[3 * i + 2], s.p[3 * k], s.p[3 * k + 1],
                                                 s.p[3 * k + 2]));
            }
        if (__any_sync(0xffffffffu, m < INFINITY))
            for (int o = 16; o > 0; o >>= 1) m = fmin(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) s.wmin[warp] = m;
        // trials of this sweep (each sphere draws 4 uniforms, the fourth is unused)
        const uint64_t cbase = (uint64_t)sweep * 4 * (uint64_t)n;   // counters used before this sweep
        for (int i = t; i < n; i += kThreads) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const double u = uniform(base, cbase + 4 * (uint64_t)i + a + 1);
                const double mv = __dmul_rn(step, __dsub_rn(__dmul_rn(2.0, u), 1.0));
                s.tr[3 * i + a] = wrap1(__dadd_rn(s.p[3 * i + a], mv));
            }
            s.tf[i] = narrow(s.tr[3 * i], s.tr[3 * i + 1], s.tr[3 * i + 2]);
        }
        __syncthreads();
        if (t == 0) {
            double d2 = INFINITY;
            for (int w = 0; w < kWarps; ++w)
                if (s.wmin[w] < d2) d2 = s.wmin[w];
            const double half = __dmul_rn(0.5, __dsqrt_rn(d2));
            const double r_work = half < r_target ? half : r_target;
            if (r_work >= r_target && d2 > lim_target) {
                s.done = 1;
            } else {
                const double tw = __dmul_rn(2.0, r_work);
                s.lim = __dmul_rn(tw, tw);
            }
        }
        __syncthreads();
        if (s.done) break;
        const double lim = s.lim;
        const float limf = (float)lim;
        for (int i0 = 0; i0 < n; i0 += kRows) {
            const int nr = min(kRows, n - i0), bw = (nr + 31) / 32;
            // One warp per trial: its bit rows, and whether they settle it.  A centre k that the
            // trial is not clear of rejects it unless k may have moved before (k < i in the
            // block) to a place it is clear of; a trial clear of every place that any sphere can
            // have is taken whatever happens.  Only the others depend on the order.
            if (t < kRows / 32) s.acc[t] = s.open[t] = 0;
            __syncthreads();
            for (int ri = warp; ri < nr; ri += kWarps) {
                const int i = i0 + ri;
                bool reject = false, sure = true;
                for (int w = 0; w < words && !reject; ++w) {
                    const int k = w * 32 + lane;
                    bool a = true, b = true;
                    if (k < n && k != i) a = clear_of(s.tf[i], s.pf[k], s.tr + 3 * i, s.p + 3 * k, limf, lim);
                    const bool may = k >= i0 && k < i;               // k's move of this sweep comes first
                    if (may) b = clear_of(s.tf[i], s.tf[k], s.tr + 3 * i, s.tr + 3 * k, limf, lim);
                    const unsigned wa = __ballot_sync(0xffffffffu, a), wb = __ballot_sync(0xffffffffu, b);
                    reject = __any_sync(0xffffffffu, !a && !(may && b));
                    sure = sure && __all_sync(0xffffffffu, a && b);
                    if (lane == 0) {
                        s.A[ri][w] = wa;
                        s.B[ri][w] = wb;
                    }
                }
                if (lane == 0 && !reject) atomicOr(sure ? &s.acc[ri >> 5] : &s.open[ri >> 5], 1u << (ri & 31));
            }
            __syncthreads();
            if (warp == 0) {   // the open trials in order; lane w holds word w of the rows
                const int w0 = i0 / 32;                            // the block's first word
                const bool in = lane >= w0 && lane < w0 + bw;
                unsigned acc = in ? s.acc[lane - w0] : 0u;         // trials taken, of lane's word
                for (int ow = 0; ow < bw; ++ow)
                    for (unsigned left = s.open[ow]; left; left &= left - 1) {
                        const int bit = __ffs(left) - 1, ri = 32 * ow + bit;
                        const unsigned a = lane < words ? s.A[ri][lane] : 0xffffffffu;
                        const unsigned b = lane < words ? s.B[ri][lane] : 0xffffffffu;
                        // trials taken before i (b is all ones elsewhere)
                        const unsigned before = lane < w0 + ow ? acc : (lane == w0 + ow ? acc & ((1u << bit) - 1u) : 0u);
                        const bool ok = __all_sync(0xffffffffu, ((before & b) | (~before & a)) == 0xffffffffu);
                        if (ok && lane == w0 + ow) acc |= 1u << bit;
                    }
                if (in) s.acc[lane - w0] = acc;
            }
            __syncthreads();
            for (int ri = t; ri < nr; ri += kThreads)
                if (s.acc[ri >> 5] >> (ri & 31) & 1u) {
                    const int i = i0 + ri;
                    for (int a = 0; a < 3; ++a) s.p[3 * i + a] = s.tr[3 * i + a];
                    s.pf[i] = s.tf[i];
                }
            __syncthreads();
        }
    }
    for (int i = t; i < 3 * n; i += kThreads) c[i] = s.p[i];
    if (t == 0) {
        state[0] = s.done;
        state[1] = sweep;
    }
}

}  // namespace rsa

// Device scratch of a placement: centres, counters, filter bits and survivor list.
struct PlaceScratch {
    double* c;          // 3 n
    long long* state;   // 4
    unsigned* bits;     // rsa::kChunk / 32
    int* list;          // rsa::kSurvivors
    static size_t bytes(int n) {
        return (3 * (size_t)n + 4) * sizeof(double) + rsa::kChunk / 8 + rsa::kSurvivors * sizeof(int);
    }
    PlaceScratch(void* p, int n) {
        c = static_cast<double*>(p);
        state = reinterpret_cast<long long*>(c + 3 * (size_t)n);
        bits = reinterpret_cast<unsigned*>(state + 4);
        list = reinterpret_cast<int*>(bits + rsa::kChunk / 32);
    }
};

// Runs RSA at radius r from one stream; h_state[0]: spheres placed.  False with the error set on
// a CUDA failure.
static bool run_rsa(cudaStream_t st, uint64_t seed, int stream, int n, double r, long long max_candidates,
                    const PlaceScratch& d, long long h_state[4]) {
    const uint64_t base = seed + (uint64_t)stream * rsa::kStream;
    const double tr = 2.0 * r;
    const double lim = tr * tr;
    const long long limit = (max_candidates + rsa::kBlock - 1) / rsa::kBlock * rsa::kBlock;
    cudaError_t e = cudaMemsetAsync(d.state, 0, 4 * sizeof(long long), st);
    rsa::k_rsa<<<1, rsa::kThreads, 0, st>>>(base, n, lim, 0, std::min(limit, (long long)rsa::kBlock), nullptr, 0, d.c, d.state);
    long long next = rsa::kBlock;
    for (;;) {
        if (e == cudaSuccess) e = cudaMemcpyAsync(h_state, d.state, 4 * sizeof(long long), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) {
            set_error("RSA kernel: %s", cudaGetErrorString(e));
            return false;
        }
        next += h_state[3];   // (0 after the first block)
        if (h_state[0] >= n || next >= limit) return true;
        const int count = (int)std::min((long long)rsa::kChunk, limit - next);
        rsa::k_rsa_filter<<<(count + 255) / 256, 256, 0, st>>>(base, lim, next, count, d.c, d.state, d.bits);
        rsa::k_rsa_list<<<1, rsa::kThreads, 0, st>>>(d.bits, count, d.list, d.state);
        rsa::k_rsa<<<1, rsa::kThreads, 0, st>>>(base, n, lim, 0, rsa::kSurvivors, d.list, next, d.c, d.state);
        e = cudaGetLastError();
    }
}

// The placement of steps 1-2 above into host memory (3 n centres); generator: 0 RSA,
// 1 RSA at 0.85 r + growth sweeps.
static hmg_status place(hmg_ctx* ctx, uint64_t seed, int n, double r, long long max_candidates,
                        std::vector<double>& centres, int* generator) {
    DeviceGuard dg(ctx->device);
    cudaStream_t st = ctx->stream;
    // The kept scratch holds 1024 spheres and the filter's bits and survivor list.  Like the tables of
    // the grid sizes it is a fixed part of a context, outside the budget, which is for state that grows
    // with the work: of a placement the centres and counters, counted for the call.
    const size_t bytes = (3 * (size_t)n + 2) * sizeof(double);
    const bool counted = ctx->reserve(bytes);
    void* mem = counted ? ctx->scratch_get(PlaceScratch::bytes(n)) : nullptr;
    if (!mem) {
        if (counted) ctx->unreserve(bytes);
        set_error("cannot allocate placement state");
        return HMG_OUT_OF_MEMORY;
    }
    const PlaceScratch d(mem, n);
    double* d_c = d.c;
    long long* d_state = d.state;
    long long h[4] = {0, 0, 0, 0};
    hmg_status res = HMG_OK;
    int gen = 0;
    if (!run_rsa(st, seed, 0, n, r, max_candidates, d, h)) {
        res = HMG_CUDA_ERROR;
    } else if (h[0] < n) {
        gen = 1;
        const double r85 = 0.85 * r;
        if (!run_rsa(st, seed, 2, n, r85, max_candidates, d, h)) {
            res = HMG_CUDA_ERROR;
        } else if (h[0] < n) {
            set_error("RSA at the reduced radius placed %lld of %d spheres", h[0], n);
            res = HMG_NOT_CONVERGED;
        } else if (n > 1) {
            const double tr = 2.0 * r;
            cudaFuncSetAttribute(rsa::k_grow, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(rsa::GrowSmem));
            rsa::k_grow<<<1, rsa::kThreads, sizeof(rsa::GrowSmem), st>>>(seed + 1 * rsa::kStream, n, r, tr * tr, 20000, d_c, d_state);
            cudaError_t e = cudaMemcpyAsync(h, d_state, 2 * sizeof(long long), cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            if (e != cudaSuccess) {
                set_error("growth kernel: %s", cudaGetErrorString(e));
                res = HMG_CUDA_ERROR;
            } else if (!h[0]) {
                set_error("growth sweeps did not reach the target radius in 20000 sweeps");
                res = HMG_NOT_CONVERGED;
            }
        }
    }
    if (res == HMG_OK) {
        centres.resize(3 * (size_t)n);
        cudaError_t e = cudaMemcpyAsync(centres.data(), d_c, 3 * (size_t)n * sizeof(double), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) {
            set_error("centre copy: %s", cudaGetErrorString(e));
            res = HMG_CUDA_ERROR;
        }
    }
    ctx->scratch_put(mem);
    ctx->unreserve(bytes);
    if (generator) *generator = gen;
    return res;
}

static bool check_place_args(hmg_ctx* ctx, int n, double r, long long max_candidates) {
    if (!ctx || n < 1 || n > rsa::kMaxSpheres || !(r > 0.0 && r < 0.5) || max_candidates < 1) {
        set_error("need a context, 1 <= n <= %d, 0 < r < 0.5 and a positive candidate cap", rsa::kMaxSpheres);
        return false;
    }
    return true;
}

}  // namespace hmg

using namespace hmg;

extern "C" hmg_status hmg_rsa(hmg_ctx* ctx, uint64_t seed, int n, double r, long long max_candidates,
                              hmg_sphere* spheres_out, int* generator) {
    g_last_error.clear();
    if (!check_place_args(ctx, n, r, max_candidates) || !spheres_out) {
        if (!spheres_out) set_error("null output");
        return HMG_INVALID_ARG;
    }
    std::vector<double> c;
    hmg_status st = place(ctx, seed, n, r, max_candidates, c, generator);
    if (st != HMG_OK) return st;
    std::vector<hmg_sphere> h(n);
    for (int i = 0; i < n; ++i) h[i] = hmg_sphere{c[3 * i], c[3 * i + 1], c[3 * i + 2], r};
    DeviceGuard dg(ctx->device);
    if (is_device_ptr(spheres_out)) {
        if (cudaMemcpy(spheres_out, h.data(), n * sizeof(hmg_sphere), cudaMemcpyHostToDevice) != cudaSuccess) {
            set_error("sphere copy: %s", cudaGetErrorString(cudaGetLastError()));
            return HMG_CUDA_ERROR;
        }
    } else {
        for (int i = 0; i < n; ++i) spheres_out[i] = h[i];
    }
    return HMG_OK;
}

extern "C" hmg_status hmg_rve(hmg_ctx* ctx, uint64_t seed, int n, double r, long long max_candidates, double layer,
                              int N, uint8_t* phase_out, hmg_sphere* spheres_out, int* generator) {
    g_last_error.clear();
    if (!check_place_args(ctx, n, r, max_candidates)) return HMG_INVALID_ARG;
    if (!phase_out || !valid_N(N) || !(layer > 0.0 && layer < 1.0)) {
        set_error("need a phase buffer, a valid N and a layer in (0, 1)");
        return HMG_INVALID_ARG;
    }
    std::vector<double> c;
    hmg_status st = place(ctx, seed, n, r, max_candidates, c, generator);
    if (st != HMG_OK) return st;
    std::vector<hmg_sphere> h(n);
    for (int i = 0; i < n; ++i) h[i] = hmg_sphere{c[3 * i], c[3 * i + 1], c[3 * i + 2], r};
    if (spheres_out) {
        DeviceGuard dg(ctx->device);
        if (is_device_ptr(spheres_out)) {
            if (cudaMemcpy(spheres_out, h.data(), n * sizeof(hmg_sphere), cudaMemcpyHostToDevice) != cudaSuccess) {
                set_error("sphere copy: %s", cudaGetErrorString(cudaGetLastError()));
                return HMG_CUDA_ERROR;
            }
        } else {
            for (int i = 0; i < n; ++i) spheres_out[i] = h[i];
        }
    }
    return hmg_voxelize(ctx, h.data(), (size_t)n, layer, N, phase_out);
}
