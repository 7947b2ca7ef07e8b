// libhmg host runtime: contexts, transform tables, device buffers, the solve driver of
// §3's Algorithm (FP64 and FP32-bulk with FP64 defect correction), and the C ABI.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/hmg.h"
#include "hmg_internal.h"
#include "hmg_runtime.h"

namespace hmg {

thread_local std::string g_last_error;

void set_error(const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_last_error = buf;
}

// ---------------------------------------------------------------------------
// grid sizes and twiddles
// ---------------------------------------------------------------------------

bool valid_length(int L) {
    if (L < 1) return false;
    while (L % 2 == 0) L /= 2;
    while (L % 3 == 0) L /= 3;
    return L == 1;
}

bool valid_N(int N) { return N >= 8 && N <= 512 && N % 2 == 0 && valid_length(N); }

// w_L^k = exp(-2 pi i k / L), k < L, rounded to 62 fractional bits: {re high, re low, im high,
// im low} with value high 2^-30 + low 2^-62, low signed.  Angles are reduced to the first
// octant in integers, so the symmetries of the table hold exactly.
void fixed_twiddles(int L, int4* out) {
    for (int k = 0; k < L; ++k) {
        const int oct = 8 * k / L;                                  // octant of the angle
        int r = 8 * k - oct * L;                                     // remainder, in units of (2 pi / 8) / L
        if (oct & 1) r = L - r;
        const long double ang = 0.78539816339744830961566084581988L * (long double)r / (long double)L;
        const long double c = std::cos(ang), s = std::sin(ang), one = 4611686018427387904.0L;   // 2^62
        const long long ci = std::llround(c * one), si = std::llround(s * one);
        const bool sw = ((oct + 1) & 2) != 0;                        // octants 1, 2, 5, 6
        long long re = sw ? si : ci, im = sw ? ci : si;
        if (oct >= 2 && oct < 6) re = -re;
        if (oct < 4) im = -im;                                       // forward sign
        const int rl = (int)(unsigned)(unsigned long long)re, il = (int)(unsigned)(unsigned long long)im;
        out[k] = make_int4((int)((re - rl) >> 32), rl, (int)((im - il) >> 32), il);
    }
}

GridPlan::~GridPlan() {
    if (tw32) cudaFree(tw32);
    if (twf) cudaFree(twf);
    if (rcp) cudaFree(rcp);
}

}  // namespace hmg

std::shared_ptr<hmg::GridPlan> hmg_ctx::plan(int N) {
    using namespace hmg;
    auto it = plans.find(N);
    if (it != plans.end()) return it->second;
    auto gp = std::make_shared<GridPlan>();
    gp->N = N;
    const int M = N / 2;
    std::vector<float2> h32(N + M);
    std::vector<int4> hf(N + M);
    fixed_twiddles(N, hf.data());
    fixed_twiddles(M, hf.data() + N);
    for (int part = 0; part < 2; ++part) {
        const int L = part == 0 ? N : M;
        const int off = part == 0 ? 0 : N;
        for (int k = 0; k < L; ++k) {
            // exp(-2 pi i k / L), evaluated with the octant symmetry so that
            // w^(L/4) = -i, w^(L/2) = -1 hold exactly
            const double ang = 2.0 * M_PI * (double)k / (double)L;
            double c = std::cos(ang), s = -std::sin(ang);
            if ((4 * k) % L == 0) {
                const int qd = (4 * k) / L;
                c = (qd == 0) ? 1.0 : (qd == 2 ? -1.0 : 0.0);
                s = (qd == 1) ? -1.0 : (qd == 3 ? 1.0 : 0.0);
            }
            h32[off + k] = make_float2((float)c, (float)s);
        }
    }
    if (cudaMalloc(&gp->twf, sizeof(int4) * (N + M)) != cudaSuccess ||
        cudaMalloc(&gp->rcp, sizeof(long long) * fx_rcp_count(N)) != cudaSuccess ||
        cudaMalloc(&gp->tw32, sizeof(float2) * (N + M)) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    cudaMemcpy(gp->twf, hf.data(), sizeof(int4) * (N + M), cudaMemcpyHostToDevice);
    cudaMemcpy(gp->tw32, h32.data(), sizeof(float2) * (N + M), cudaMemcpyHostToDevice);
    fx_rcp_table(gp->rcp, N);
    if (cudaStreamSynchronize(0) != cudaSuccess) {   // the table is read from other streams
        cudaGetLastError();
        return nullptr;
    }
    plans[N] = gp;
    return gp;
}

namespace hmg {

GridDesc make_desc(const GridPlan& gp, const double k[3], const uint8_t* phase_d, int* exps,
                   int nslots, int scheme, double beta) {
    GridDesc g;
    memset(&g, 0, sizeof(g));
    const int N = gp.N, M = N / 2;
    g.N = N;
    g.M = M;
    g.NN = (long long)N * N;
    g.N3 = g.NN * N;
    g.NNM = g.NN * M;
    g.tw32 = gp.tw32;
    g.twf = gp.twf;
    g.rcp = gp.rcp;
    const double kmin = std::min(k[0], std::min(k[1], k[2]));
    const double kmax = std::max(k[0], std::max(k[1], k[2]));
    g.scheme = scheme;
    if (scheme == HMG_SCHEME_BASIC) {
        // basic scheme: positive reference medium at the centre of the conductivity range,
        // e^{n+1} = E - Gamma0 * ((k - k0) e^n) with Gamma0 = P / k0, on the field e itself
        const double k0 = 0.5 * (kmin + kmax);
        g.k0 = k0;
        for (int p = 0; p < 3; ++p) {
            g.Y[p] = (k[p] - k0) / k0;
            g.W[p] = k[p];
            g.KP[p] = 1.0;
        }
        g.ga = 0.0;
        g.gb = 1.0;
        g.gc = 1.0;
        g.epsf = 1.0;
    } else {
        // Eyre-Milton (tau = (k + k0) e): tau^{n+1} = (I - 2P)(Y tau^n) + 2 k0 E.  The
        // augmented Lagrangian scheme (beta = 1) and the relaxed polarization iteration
        // keep a fraction of the old field: tau^{n+1} = (1 - beta/2) tau^n + (beta/2) T tau^n,
        // whose step moves beta/2 of the Eyre-Milton step, so the step-6 residual
        // |e^n - e_comp^n| = |T tau^n - tau^n| / (2 k0) is |tau^{n+1} - tau^n| / (beta k0).
        if (scheme == HMG_SCHEME_AUGMENTED_LAGRANGIAN) beta = 1.0;
        const double k0 = std::sqrt(kmin * kmax);
        g.k0 = k0;
        for (int p = 0; p < 3; ++p) {
            g.Y[p] = (k[p] - k0) / (k[p] + k0);
            g.W[p] = k[p] / (k[p] + k0);
            g.KP[p] = k[p] + k0;
        }
        g.ga = 1.0;
        g.gb = 2.0;
        g.gc = 2.0 * k0;
        g.relax = 1.0 - 0.5 * beta;
        g.epsf = 1.0 / (beta * k0);
    }
    for (int p = 0; p < 3; ++p) g.YN[p] = std::ldexp(g.Y[p] * (1.0 / (double)g.N3), scale_bits(N));
    for (int s = 0; s < kMaxSlots; ++s)
        for (int c = 0; c < 3; ++c) g.E[s][c] = (s == c) ? 1.0 : 0.0;
    g.nslots = nslots;
    g.comps = 3;
    g.expA = exps;
    g.expB = exps ? exps + 3 * (size_t)nslots * g.NN : nullptr;
    g.phase = phase_d;
    return g;
}

static float time_launches(cudaStream_t st, const std::function<void()>& f, int reps) {
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    f();   // warm-up
    cudaEventRecord(a, st);
    for (int r = 0; r < reps; ++r) f();
    cudaEventRecord(b, st);
    cudaEventSynchronize(b);
    float ms = 1e30f;
    if (cudaEventElapsedTime(&ms, a, b) != cudaSuccess) ms = 1e30f;
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    return ms;
}

// On-disk record of the autotuner's choices, opt-in through the environment variable
// HMG_TUNE_CACHE (a file path): one line "<device name>|<SM count>|<N>|<variant>" per
// choice, the last line for a key wins.  A context takes a recorded choice for its GPU
// instead of timing the variants, and appends what it times.
namespace {
std::mutex g_tune_mu;

std::string tune_key(int device, int N) {
    cudaDeviceProp p;
    if (cudaGetDeviceProperties(&p, device) != cudaSuccess) {
        cudaGetLastError();
        return std::string();
    }
    return std::string(p.name) + "|" + std::to_string(p.multiProcessorCount) + "|" + std::to_string(N) + "|";
}

bool tune_cache_read(int device, int N, int* variant) {
    const char* path = std::getenv("HMG_TUNE_CACHE");
    if (!path || !*path) return false;
    const std::string key = tune_key(device, N);
    if (key.empty()) return false;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    FILE* f = std::fopen(path, "r");
    if (!f) return false;
    char line[512];
    bool found = false;
    while (std::fgets(line, sizeof line, f)) {
        const std::string l(line);
        if (l.compare(0, key.size(), key) != 0) continue;
        const int v = std::atoi(l.c_str() + key.size());
        if (v >= 0 && v < 32 && !(v & 4)) {
            *variant = v;
            found = true;
        }
    }
    std::fclose(f);
    return found;
}

void tune_cache_write(int device, int N, int variant) {
    const char* path = std::getenv("HMG_TUNE_CACHE");
    if (!path || !*path) return;
    const std::string key = tune_key(device, N);
    if (key.empty()) return;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    if (FILE* f = std::fopen(path, "a")) {
        std::fprintf(f, "%s%d\n", key.c_str(), variant);
        std::fclose(f);
    }
}
}  // namespace

int autotune_z(::hmg_ctx* c, GridDesc g, SolveState* s, cudaStream_t st) {
    auto it = c->ztune.find(g.N);
    if (it != c->ztune.end()) return it->second;
    int best = 0;
    if (tune_cache_read(c->device, g.N, &best)) {
        c->ztune[g.N] = best;
        return best;
    }
    if (!s->spec32 || !s->f32buf) {
        c->ztune[g.N] = best;
        return best;
    }
    const unsigned all = (1u << g.nslots) - 1u;
    const size_t bytes = (size_t)g.nslots * 3 * g.N3 * sizeof(float);
    cudaMemsetAsync(s->spec32, 0, bytes, st);
    cudaMemsetAsync(s->f32buf, 0, bytes, st);
    // z pass: two kernels
    int zbest = 0, zpbest = 0;
    if (fast_z_ctas(g)) {
        // three z kernels: components in one thread, per-component groups, and the first
        // as a persistent kernel with staged columns
        float zms[3];
        for (int v = 0; v < 3; ++v) {
            g.zvar = v == 1 ? 1 : 0;
            g.zpers = v == 2 ? 1 : 0;
            zms[v] = time_launches(st, [&] { launch_z_pass<float>(g, Z_ITER, all, s->spec32, nullptr, st); }, 4);
        }
        int b = 0;
        for (int v = 1; v < 3; ++v)
            if (zms[v] < zms[b]) b = v;
        if (b == 2 && fast_take_wait_failure()) b = 0;
        zbest = b == 1 ? 1 : 0;
        zpbest = b == 2 ? 1 : 0;
        g.zpers = 0;
    }
    // x and y passes: fused cluster kernels or separate passes
    int xybest = 0;
    if (fused_cluster(g.N)) {
        float xyms[2];
        for (int v = 0; v < 2; ++v) {
            g.xyvar = v;
            xyms[v] = time_launches(st, [&] {
                if (v == 0 && fast_x_ctas(g)) {   // separate passes: a chained sweep's x and y work
                    launch_y_pass<float>(g, true, all, s->spec32, st);
                    launch_y_pass<float>(g, false, all, s->spec32, st);
                    fast_x_round(g, false, false, all, s->spec32, s->f32buf, nullptr, st);
                    return;
                }
                launch_xy_forward<float>(g, XF_POLARIZE, all, s->f32buf, s->spec32, nullptr, st);
                launch_yx_inverse<float>(g, XI_INPLACE, all, s->spec32, s->f32buf, nullptr, nullptr, nullptr, nullptr, st);
            }, 3);
        }
        xybest = xyms[1] < xyms[0] ? 1 : 0;
    }
    // chained x round trip: the plain kernel or the persistent one with staged rows
    int xpbest = 0;
    g.zvar = zbest;
    g.xyvar = xybest;
    if (chain_sweeps(g) && fast_x_ctas(g)) {
        float xms[2];
        for (int v = 0; v < 2; ++v) {
            g.xpers = v;
            xms[v] = time_launches(st, [&] { fast_x_round(g, false, false, all, s->spec32, s->f32buf, nullptr, st); }, 6);
        }
        xpbest = xms[1] < xms[0] ? 1 : 0;
        if (fast_take_wait_failure()) xpbest = 0;
    }
    cudaGetLastError();
    // bit 5 (the plane kernel) is not timed here: alone it times a few per cent faster than
    // the three passes it replaces, inside a solve it is even, so it is left to hmg_set_variant
    best = zbest | (xybest << 1) | (xpbest << 3) | (zpbest << 4);
    c->ztune[g.N] = best;
    tune_cache_write(c->device, g.N, best);
    return best;
}

// ---------------------------------------------------------------------------
// device buffers
// ---------------------------------------------------------------------------

}  // namespace hmg

bool hmg_ctx::reserve(size_t bytes) {
    size_t cur = pool->used.load();
    do {
        if (pool->limit && cur + bytes > pool->limit) return false;
    } while (!pool->used.compare_exchange_weak(cur, cur + bytes));
    return true;
}

void hmg_ctx::unreserve(size_t bytes) { pool->used -= bytes; }

void* hmg_ctx::alloc(size_t bytes) {
    if (bytes == 0) return nullptr;
    // reserve the bytes in the (possibly shared) budget first
    if (!reserve(bytes)) return nullptr;
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) != cudaSuccess) {
        cudaGetLastError();
        unreserve(bytes);
        return nullptr;
    }
    sizes[p] = bytes;
    return p;
}

void hmg_ctx::release(void* p) {
    if (!p) return;
    auto it = sizes.find(p);
    if (it != sizes.end()) {
        pool->used -= it->second;
        sizes.erase(it);
    }
    cudaFree(p);
}

void* hmg_ctx::scratch_get(size_t bytes) {
    if (bytes <= kScratchBytes && scratch) return scratch;
    void* p = nullptr;
    if (cudaMalloc(&p, bytes <= kScratchBytes ? kScratchBytes : bytes) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    if (bytes <= kScratchBytes) scratch = p;
    return p;
}

void hmg_ctx::scratch_put(void* p) {
    if (p && p != scratch) cudaFree(p);
}

namespace hmg {

size_t state_bytes(int N, bool fp64, int nslots) {
    const size_t N3 = (size_t)N * N * N;
    const size_t field64 = (size_t)nslots * 3 * N3 * 8;
    const size_t field32 = (size_t)nslots * 3 * N3 * 4;
    size_t b = N3 + 2 * field64;                        // phase, tau64, spec64
    if (!fp64) b += 3 * field32;                        // f32, r32, spec32
    b += (size_t)nslots * 3 * 4 * (3 * (size_t)N * N) * 8 + 4096;   // partials, FP64 exponents
    return b;
}

bool SolveState::ensure(Context* c, int N_, bool fp64_, int nslots_) {
    // a bulk (FP32 + FP64) state also serves FP64 requests
    if (N == N_ && (fp64 == fp64_ || (fp64_ && !fp64)) && nslots >= nslots_) return true;
    free_all(c);
    N = N_;
    fp64 = fp64_;
    nslots = nslots_;
    const size_t N3 = (size_t)N * N * N;
    const size_t f64 = (size_t)nslots * 3 * N3 * 8, f32 = (size_t)nslots * 3 * N3 * 4;
    phase = (uint8_t*)c->alloc(N3);
    tau64 = (double*)c->alloc(f64);
    spec64 = c->alloc(f64);
    exps = (int*)c->alloc((size_t)nslots * 6 * N * N * sizeof(int));
    if (!fp64) {
        f32buf = (float*)c->alloc(f32);
        r32 = (float*)c->alloc(f32);
        spec32 = c->alloc(f32);
    }
    const size_t np = (size_t)nslots * 3 * 3 * N * N + 64;   // at least one double per row
    partial = (double*)c->alloc(np * sizeof(double));
    partial2 = (double*)c->alloc(np * sizeof(double));
    partial3 = (double*)c->alloc(np * sizeof(double));
    red = (double*)c->alloc(kRedDoubles * sizeof(double));
    bool ok = phase && tau64 && spec64 && exps && partial && partial2 && partial3 && red &&
              (fp64 || (f32buf && r32 && spec32));
    if (!ok) {
        free_all(c);
        return false;
    }
    return true;
}

void SolveState::free_all(Context* c) {
    for (void** p : {(void**)&phase, (void**)&tau64, &spec64, (void**)&exps, (void**)&f32buf, (void**)&r32, &spec32,
                     (void**)&partial, (void**)&partial2, (void**)&partial3, (void**)&red}) {
        c->release(*p);
        *p = nullptr;
    }
    N = 0;
}

void SolveState::free_pinned() {
    if (pin) cudaFreeHost(pin);
    pin = nullptr;
}

bool SolveState::pinned() {
    if (!pin && cudaMallocHost(&pin, (kRedDoubles + 8) * sizeof(double)) != cudaSuccess) {
        cudaGetLastError();
        pin = nullptr;
        set_error("cannot allocate pinned host memory");
    }
    return pin != nullptr;
}

// ---------------------------------------------------------------------------
// pointer helpers
// ---------------------------------------------------------------------------

bool is_device_ptr(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

cudaError_t copy_in(void* dst_dev, const void* src, size_t bytes, cudaStream_t st) {
    return cudaMemcpyAsync(dst_dev, src, bytes, is_device_ptr(src) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, st);
}

cudaError_t copy_out(void* dst, const void* src_dev, size_t bytes, cudaStream_t st) {
    return cudaMemcpyAsync(dst, src_dev, bytes, is_device_ptr(dst) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, st);
}

// ---------------------------------------------------------------------------
// one sweep of steps 2-7 and the step-1 equilibrium check
// ---------------------------------------------------------------------------

int Tracer::begin(cudaStream_t st) {
    if (!on) return -1;
    int idx;
    if (!free_pairs.empty()) {
        idx = free_pairs.back();
        free_pairs.pop_back();
    } else {
        cudaEvent_t a, b;
        if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) {
            cudaGetLastError();
            return -1;
        }
        idx = (int)events.size() / 2;
        events.push_back(a);
        events.push_back(b);
    }
    cudaEventRecord(events[2 * idx], st);
    return idx;
}

void Tracer::end(int ev, int kind, double b, cudaStream_t st) {
    if (ev < 0) return;
    cudaEventRecord(events[2 * ev + 1], st);
    pending.push_back({kind, ev, b, sweep});
}

void Tracer::collect(const double* share) {
    for (const Pending& p : pending) {
        float t = 0.f;
        if (cudaEventElapsedTime(&t, events[2 * p.ev], events[2 * p.ev + 1]) == cudaSuccess) {
            ms[p.kind] += t;
            launches[p.kind] += 1;
            bytes[p.kind] += share && p.sweep >= 0 ? share[p.sweep] * p.bytes : p.bytes;
        } else {
            cudaGetLastError();
        }
        free_pairs.push_back(p.ev);
    }
    pending.clear();
}

void Tracer::reset() {
    collect();
    for (int k = 0; k < HMG_K_COUNT; ++k) {
        ms[k] = 0;
        launches[k] = 0;
        bytes[k] = 0;
    }
}

Tracer::~Tracer() {
    for (cudaEvent_t e : events) cudaEventDestroy(e);
}

static int popc(unsigned m) { return __builtin_popcount(m); }

// Each launch is bracketed by tracer events when tracing is on.
#define HMG_TRACED(KIND, BYTES, CALL)          \
    do {                                       \
        int ev_ = tr ? tr->begin(st) : -1;     \
        CALL;                                  \
        if (tr) tr->end(ev_, KIND, BYTES, st); \
    } while (0)

// FP64 launches are traced as one kind of their own.
template <typename R>
static constexpr int kind_of(int k) {
    return std::is_same<R, double>::value ? HMG_K_FP64 : k;
}

template <typename R>
void Solver::sweep(unsigned mask, R* field, void* spec, int zmode, int ximode, const float* r32in,
                   float* d32, float* r32out, double* sums, const StopRule& stop) {
    const double f = (double)popc(mask) * 3.0 * (double)g.N3;   // field elements moved per array
    const double F = sizeof(R);
    const bool fused = std::is_same<R, float>::value && g.xyvar == 1 && fused_cluster(g.N) != 0;
    double* pb = psweep ? psweep : s->partial;
    double xb = f * 2 * F;                                       // spectrum in, field out
    if (ximode == XI_INPLACE_RES) xb += f * F;                  // old field for the residual
    if (ximode == XI_ADD_R_RES) xb += f * F + f * 4;            // old field and r
    if (ximode == XI_ADD_R) xb += f * 4;                         // r
    if (ximode == XI_DIFF) xb = f * F + f * F + 2 * f * 4;      // spectrum, old field, d and r out
    if (fused) {
        // x+y forward and y+x inverse: one cluster kernel each
        HMG_TRACED(kind_of<R>(HMG_K_X_FORWARD), f * 2 * F + (double)g.N3,
                   launch_xy_forward<R>(g, XF_POLARIZE, mask, field, spec, nullptr, st));
        HMG_TRACED(kind_of<R>(HMG_K_Z_GREEN), f * 2 * F, launch_z_pass<R>(g, zmode, mask, spec, nullptr, st));
        HMG_TRACED(kind_of<R>(HMG_K_X_INVERSE), xb,
                   launch_yx_inverse<R>(g, ximode, mask, spec, field, r32in, d32, r32out, pb, st));
    } else {
        HMG_TRACED(kind_of<R>(HMG_K_X_FORWARD), f * 2 * F + (double)g.N3,
                   launch_x_forward<R>(g, XF_POLARIZE, mask, field, spec, nullptr, st));
        HMG_TRACED(kind_of<R>(HMG_K_Y_FORWARD), f * 2 * F, launch_y_pass<R>(g, true, mask, spec, st));
        HMG_TRACED(kind_of<R>(HMG_K_Z_GREEN), f * 2 * F, launch_z_pass<R>(g, zmode, mask, spec, nullptr, st));
        HMG_TRACED(kind_of<R>(HMG_K_Y_INVERSE), f * 2 * F, launch_y_pass<R>(g, false, mask, spec, st));
        HMG_TRACED(kind_of<R>(HMG_K_X_INVERSE), xb,
                   launch_x_inverse<R>(g, ximode, mask, spec, field, r32in, d32, r32out, pb, st));
    }
    if (ximode == XI_INPLACE_RES || ximode == XI_ADD_R_RES || ximode == XI_DIFF)
        HMG_TRACED(kind_of<R>(HMG_K_OTHER), 0.0, launch_reduce(pb, g.nslots, x_ctas_for<R>(g), 1, sums, st, stop));
}

template <typename R>
void Solver::sweeps(unsigned mask, R* field, void* spec, int n, double* sums, int stride, const StopRule& stop) {
    constexpr bool f64 = std::is_same<R, double>::value;
    // The FP64 round trip pays where field and spectrum stay in L2 (kernels alone, us, two passes
    // against one: 32^3 19 and 12, 72^3 86 and 55, one gradient at 128^3 140 and 94); beyond it
    // reads and writes of one more array per kernel cost what they save (96^3 163 and 162,
    // 192^3 357 and 360, 256^3 709 and 974).
    const bool in_l2 = g.nslots * 3 * (double)g.N3 * sizeof(double) <= 56e6;
    if (g.relax != 0.0 || (f64 ? !in_l2 : !fast_x_round_res_available(g))) {
        for (int b = 0; b < n; ++b) {
            if (tr) tr->sweep = b;
            sweep<R>(mask, field, spec, Z_ITER, XI_INPLACE_RES, nullptr, nullptr, nullptr, sums + b * stride, stop);
        }
        if (tr) tr->sweep = -1;
        return;
    }
    const double f = (double)popc(mask) * 3.0 * (double)g.N3, F = sizeof(R);   // field elements moved per array
    double* pb = psweep ? psweep : s->partial;
    for (int b = 0; b < n; ++b) {
        if (tr) tr->sweep = b;
        if (b == 0)
            HMG_TRACED(kind_of<R>(HMG_K_X_FORWARD), f * 2 * F + (double)g.N3,
                       launch_x_forward<R>(g, XF_POLARIZE, mask, field, spec, nullptr, st));
        HMG_TRACED(kind_of<R>(HMG_K_Y_FORWARD), f * 2 * F, launch_y_pass<R>(g, true, mask, spec, st));
        HMG_TRACED(kind_of<R>(HMG_K_Z_GREEN), f * 2 * F, launch_z_pass<R>(g, Z_ITER, mask, spec, nullptr, st));
        HMG_TRACED(kind_of<R>(HMG_K_Y_INVERSE), f * 2 * F, launch_y_pass<R>(g, false, mask, spec, st));
        if (b == n - 1) {
            HMG_TRACED(kind_of<R>(HMG_K_X_INVERSE), f * 3 * F,
                       launch_x_inverse<R>(g, XI_INPLACE_RES, mask, spec, field, nullptr, nullptr, nullptr, pb, st));
        } else if constexpr (f64) {
            HMG_TRACED(HMG_K_FP64, f * 4 * F + (double)g.N3, fx_x_round(g, mask, spec, field, pb, st));
        } else {
            HMG_TRACED(HMG_K_X_ROUND, f * 4 * F + (double)g.N3, fast_x_round_res(g, mask, spec, field, pb, st));
        }
        HMG_TRACED(kind_of<R>(HMG_K_OTHER), 0.0,
                   launch_reduce(pb, g.nslots, x_ctas_for<R>(g), 1, sums + b * stride, st, stop));
    }
    if (tr) tr->sweep = -1;
}

bool Solver::chained() const { return chain_sweeps(g); }

void Solver::block_sweep(unsigned mask, int b, int blk, int zmode, bool addr, const float* r32in, int red_off) {
    const bool last = b == blk - 1;
    const int ximode = addr ? (last ? XI_ADD_R_RES : XI_ADD_R) : (last ? XI_INPLACE_RES : XI_INPLACE);
    if (!chained()) {
        sweep<float>(mask, s->f32buf, s->spec32, zmode, ximode, r32in, nullptr, nullptr, sums() + red_off);
        return;
    }
    const double f = (double)popc(mask) * 3.0 * (double)g.N3;   // field elements moved per array
    const double F = sizeof(float);
    double* pb = psweep ? psweep : s->partial;
    // with the plane kernel, the y forward of sweeps after the first was done by the
    // previous sweep's plane kernel
    const bool yxy = g.yxy && fast_yxy_available(g);
    if (b == 0)
        HMG_TRACED(HMG_K_X_FORWARD, f * 2 * F + (double)g.N3,
                   launch_x_forward<float>(g, XF_POLARIZE, mask, s->f32buf, s->spec32, nullptr, st));
    if (b == 0 || !yxy) HMG_TRACED(HMG_K_Y_FORWARD, f * 2 * F, launch_y_pass<float>(g, true, mask, s->spec32, st));
    HMG_TRACED(HMG_K_Z_GREEN, f * 2 * F, launch_z_pass<float>(g, zmode, mask, s->spec32, nullptr, st));
    if (!last) {
        const bool wtau = b == blk - 2;   // the field the residual sweep compares against
        const double xb = f * 2 * F + (double)g.N3 + (wtau ? f * F : 0.0) + (addr ? f * F : 0.0);
        if (yxy) {
            HMG_TRACED(HMG_K_YXY, xb, fast_yxy(g, addr, wtau, mask, s->spec32, s->f32buf, r32in, st));
            return;
        }
        HMG_TRACED(HMG_K_Y_INVERSE, f * 2 * F, launch_y_pass<float>(g, false, mask, s->spec32, st));
        HMG_TRACED(HMG_K_X_ROUND, xb, fast_x_round(g, addr, wtau, mask, s->spec32, s->f32buf, r32in, st));
        return;
    }
    HMG_TRACED(HMG_K_Y_INVERSE, f * 2 * F, launch_y_pass<float>(g, false, mask, s->spec32, st));
    const double xb = f * 3 * F + (addr ? f * F : 0.0);   // spectrum and old field in, field out
    HMG_TRACED(HMG_K_X_INVERSE, xb,
               launch_x_inverse<float>(g, ximode, mask, s->spec32, s->f32buf, r32in, nullptr, nullptr, pb, st));
    HMG_TRACED(HMG_K_OTHER, 0.0, launch_reduce(pb, g.nslots, x_ctas_for<float>(g), 1, sums() + red_off, st));
}

template <typename R>
void Solver::equilibrium(unsigned mask, const R* field, void* spec) {
    const double f = (double)popc(mask) * 3.0 * (double)g.N3;
    const double F = sizeof(R);
    const bool fused = std::is_same<R, float>::value && g.xyvar == 1 && fused_cluster(g.N) != 0;
    double* pb = pflux ? pflux : s->partial;
    if (fused) {
        HMG_TRACED(kind_of<R>(HMG_K_EQ_X), f * 2 * F + (double)g.N3, launch_xy_forward<R>(g, XF_FLUX, mask, field, spec, pb, st));
    } else {
        HMG_TRACED(kind_of<R>(HMG_K_EQ_X), f * 2 * F + (double)g.N3, launch_x_forward<R>(g, XF_FLUX, mask, field, spec, pb, st));
    }
    HMG_TRACED(kind_of<R>(HMG_K_OTHER), 0.0, launch_reduce(pb, g.nslots, x_ctas_for<R>(g), 3, sums() + 16, st));
    if (!fused) HMG_TRACED(kind_of<R>(HMG_K_Y_FORWARD), f * 2 * F, launch_y_pass<R>(g, true, mask, spec, st));
    HMG_TRACED(kind_of<R>(HMG_K_EQ_Z), f * F, launch_z_pass<R>(g, Z_EQ, mask, spec, s->partial2, st));
    HMG_TRACED(kind_of<R>(HMG_K_OTHER), 0.0, launch_reduce(s->partial2, g.nslots, z_ctas_for<R>(g), 1, sums() + 32, st));
}

bool Solver::fetch(double* h, int off, int count) {
    cudaError_t e = cudaSuccess;
    if (!host) e = cudaMemcpyAsync(h, s->red + off, count * sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        set_error("CUDA error: %s", cudaGetErrorString(e));
        return false;
    }
    if (host) memcpy(h, host + off, count * sizeof(double));
    if (tr) tr->collect();
    return true;
}

// eps_comp from the sum of squared differences of the stored field between two sweeps:
// |e^n - e_comp^n| = |dtau| / (2 k0) for Eyre-Milton, = |de| for the basic scheme
// (its new iterate is e_comp^n)
double Solver::eps_from_sum(double sum, int slot) const {
    const double nE = std::sqrt(g.E[slot][0] * g.E[slot][0] + g.E[slot][1] * g.E[slot][1] +
                                g.E[slot][2] * g.E[slot][2]);
    return std::sqrt(sum / (double)g.N3) * g.epsf / nE;
}

// Smallest sum whose eps_comp is not below tol: every rounded operation of eps_from_sum is
// monotone, so one threshold on the sum gives the same decisions without a root and two
// divisions in the reduction kernel.  Bisection over the bit patterns of positive doubles.
double Solver::least_sum(double tol, int slot) const {
    uint64_t lo = 0, hi = 0x7ff0000000000000ull;   // eps(lo) < tol <= eps(hi)
    while (hi - lo > 1) {
        const uint64_t mid = lo + (hi - lo) / 2;
        double x;
        memcpy(&x, &mid, sizeof x);
        if (eps_from_sum(x, slot) < tol) lo = mid;
        else hi = mid;
    }
    double x;
    memcpy(&x, &hi, sizeof x);
    return x;
}

// eq check of the slots in `mask`; fills eps_eq and the mean flux <k e>
template <typename R>
bool Solver::check_eq(unsigned mask, const R* field, void* spec, double eps_eq[3], double flux[3][3]) {
    equilibrium<R>(mask, field, spec);
    double h[48];
    if (!fetch(h, 16, 32)) return false;
    for (int sl = 0; sl < g.nslots; ++sl) {
        if (!((mask >> sl) & 1u)) continue;
        double nrm = 0.0;
        for (int c = 0; c < 3; ++c) {
            flux[sl][c] = h[sl * 3 + c] / (double)g.N3;
            nrm += flux[sl][c] * flux[sl][c];
        }
        eps_eq[sl] = std::sqrt(h[16 + sl]) / std::sqrt(nrm);
    }
    return true;
}

// Plain FP64 method: the Algorithm of §3 in its printed order, per gradient.  Up to kAhead64
// sweeps are launched before the host looks at their residuals: the reduction of each residual
// clears its gradient's flag on the device when step 1 is due (or the residual is not a
// number), and the sweeps behind it skip that gradient.  Every gradient goes through the
// sequence of sweeps and tests that one look per sweep would give.
hmg_status Solver::run_fp64(int max_iter, double tol, hmg_info* info, double K[9]) {
    host = s->pin;
    const unsigned all = (1u << g.nslots) - 1u;
    HMG_TRACED(HMG_K_OTHER, 0.0, launch_init_tau<double>(g, all, s->tau64, st));
    double eps_comp[3] = {INFINITY, INFINITY, INFINITY}, eps_eq[3] = {INFINITY, INFINITY, INFINITY};
    double flux[3][3] = {};
    int iters[3] = {0, 0, 0}, status[3] = {HMG_NOT_CONVERGED, HMG_NOT_CONVERGED, HMG_NOT_CONVERGED};
    unsigned active = max_iter > 0 ? all : 0u;
    StopRule stop;
    stop.flags = reinterpret_cast<int*>(s->red + 56);
    for (int sl = 0; sl < g.nslots; ++sl) stop.least[sl] = least_sum(tol, sl);
    Solver ahead = *this;
    ahead.g.dflags = stop.flags;
    const double* h = s->pin + 64;                                // sums of the block's sweeps
    int* hf = reinterpret_cast<int*>(s->pin + kRedDoubles);       // flags as set before the block
    double rate = 0.0;                                            // last contraction per sweep
    while (active) {
        unsigned eqm = 0;
        for (int sl = 0; sl < g.nslots; ++sl)
            if (((active >> sl) & 1u) && eps_comp[sl] < tol) eqm |= 1u << sl;
        if (eqm) {  // step 1
            if (!check_eq<double>(eqm, s->tau64, s->spec64, eps_eq, flux)) return HMG_CUDA_ERROR;
            for (int sl = 0; sl < g.nslots; ++sl)
                if (((eqm >> sl) & 1u) && eps_eq[sl] < tol) {
                    status[sl] = HMG_OK;
                    active &= ~(1u << sl);
                }
            if (!active) break;
        }
        // sweeps to launch: as many as the slowest gradient still seems to need
        int blk = 1;
        for (int sl = 0; sl < g.nslots; ++sl) {
            hf[sl] = (active >> sl) & 1u ? SF_ACTIVE : 0;
            if (!hf[sl]) continue;
            double need = kAhead64;
            if (std::isfinite(eps_comp[sl]) && rate > 0.0 && rate < 1.0)
                need = eps_comp[sl] > tol ? std::ceil(std::log(tol / eps_comp[sl]) / std::log(rate)) : 1.0;
            blk = std::max(blk, (int)std::min((double)kAhead64, need));
        }
        for (int sl = 0; sl < g.nslots; ++sl)
            if ((active >> sl) & 1u) blk = std::min(blk, max_iter - iters[sl]);
        cudaMemcpyAsync(stop.flags, hf, 3 * sizeof(int), cudaMemcpyHostToDevice, st);
        ahead.sweeps<double>(active, s->tau64, s->spec64, blk, s->pin + 64, 3, stop);
        const cudaError_t ce = cudaStreamSynchronize(st);
        if (ce != cudaSuccess) {
            set_error("CUDA error: %s", cudaGetErrorString(ce));
            return HMG_CUDA_ERROR;
        }
        if (tr) {   // bytes of the gradients whose sweep was not skipped
            double share[kAhead64] = {};
            for (int b = 0; b < blk; ++b)
                for (int sl = 0; sl < g.nslots; ++sl)
                    if (((active >> sl) & 1u) && !(h[3 * b + sl] < 0.0)) share[b] += 1.0 / popc(active);
            tr->collect(share);
        }
        for (int sl = 0; sl < g.nslots; ++sl) {
            if (!((active >> sl) & 1u)) continue;
            for (int b = 0; b < blk; ++b) {
                if (h[3 * b + sl] < 0.0) break;   // stopped at the sweep before
                const double before = eps_comp[sl];
                ++iters[sl];
                eps_comp[sl] = eps_from_sum(h[3 * b + sl], sl);
                if (std::isfinite(before) && before > 0.0) rate = eps_comp[sl] / before;
            }
            if (!std::isfinite(eps_comp[sl])) {
                status[sl] = HMG_DIVERGED;
                active &= ~(1u << sl);
            } else if (iters[sl] >= max_iter) {
                active &= ~(1u << sl);   // out of sweeps
            }
        }
    }
    // slots that ran out of sweeps: report the last iterate
    unsigned left = 0;
    for (int sl = 0; sl < g.nslots; ++sl)
        if (status[sl] == HMG_NOT_CONVERGED) left |= 1u << sl;
    if (left && !check_eq<double>(left, s->tau64, s->spec64, eps_eq, flux)) return HMG_CUDA_ERROR;
    return finish(status, iters, iters, eps_comp, eps_eq, flux, 0, info, K);
}

// FP32 bulk: FP32 sweeps until the FP32 residual stalls, then FP64 defect correction
// rounds: r = T tau64 + b - tau64 (one FP64 sweep), the FP64 equilibrium test when the
// FP64 residual is below tol, FP32 sweeps on delta = T delta + r, tau64 += delta, until
// the FP64 residuals meet the tolerance.  Each tick launches the FP64 work of the
// gradients that need it on a second stream, next to a block of FP32 sweeps of the
// others (FP64 arithmetic and HBM traffic overlap); the FP64 equilibrium test of a
// gradient runs in the tick after its FP64 sweep.  Each gradient goes through the
// same sequence of operations whatever the others do.
hmg_status Solver::run_bulk(int max_iter, double tol, hmg_info* info, double K[9], cudaStream_t st64) {
    enum { PH_A = 0, PH_OUTER = 1, PH_EQ = 2, PH_INNER = 3, PH_DONE = 4 };
    const unsigned all = (1u << g.nslots) - 1u;
    HMG_TRACED(HMG_K_OTHER, 0.0, launch_init_tau<float>(g, all, s->f32buf, st));
    int state[3], iters[3] = {0, 0, 0}, it64[3] = {0, 0, 0}, status[3];
    double eps_comp[3] = {INFINITY, INFINITY, INFINITY}, eps_eq[3] = {INFINITY, INFINITY, INFINITY};
    double eps32[3] = {INFINITY, INFINITY, INFINITY}, best[3], outer_eps[3] = {INFINITY, INFINITY, INFINITY};
    double qeq[3];   // the ratio eps_eq / eps_comp the correction solves aim for
    int since_best[3] = {0, 0, 0};
    double flux[3][3] = {};
    int rounds = 0;
    for (int sl = 0; sl < 3; ++sl) {
        state[sl] = sl < g.nslots ? PH_A : PH_DONE;
        status[sl] = HMG_NOT_CONVERGED;
        best[sl] = INFINITY;
    }
    const bool em = g.scheme == HMG_SCHEME_EYRE_MILTON && g.relax == 0.0;
    const double thetaA = std::max(tol, em ? kBulkExit : kBulkExitSlow);
    for (int sl = 0; sl < 3; ++sl) qeq[sl] = em ? kEqRatio0 : kEqRatio0Slow;
    const double eta = 1e-4;           // inner solves reduce the outer residual by this factor
    const int stall = 24;              // sweeps without a new best residual = FP32 floor
    // a new best must improve by this factor; the basic scheme contracts by only
    // rho = max|Y| = (c - 1) / (c + 1) per sweep, so its bar follows rho
    double rho = 0.0;
    for (int p = 0; p < 3; ++p) rho = std::max(rho, std::fabs(g.Y[p]));
    const double improve = g.scheme == HMG_SCHEME_BASIC
                               ? std::min(0.999, 1.0 - 0.25 * (1.0 - std::pow(rho, (double)kResidualEvery)))
                               : 0.999;
    auto mask_of = [&](int ph) {
        unsigned m = 0;
        for (int sl = 0; sl < g.nslots; ++sl)
            if (state[sl] == ph) m |= 1u << sl;
        return m;
    };
    host = s->pin;
    Solver s64{g, s, st64, tr, s->partial3, s->partial3, s->pin};
    cudaEvent_t ready;
    if (cudaEventCreateWithFlags(&ready, cudaEventDisableTiming) != cudaSuccess) {
        set_error("event create failed");
        return HMG_CUDA_ERROR;
    }
    const double* h = s->pin;
    int total = 0;
    hmg_status err = HMG_OK;
    while (mask_of(PH_DONE) != all && total < max_iter) {
        ++total;
        // FP64 work on the second stream, after this stream's pending transitions
        const unsigned me = mask_of(PH_EQ), mo = mask_of(PH_OUTER);
        if (me || mo) {
            cudaEventRecord(ready, st);
            cudaStreamWaitEvent(st64, ready, 0);
        }
        if (me) s64.equilibrium<double>(me, s->tau64, s->spec64);
        if (mo) s64.sweep<double>(mo, s->tau64, s->spec64, Z_ITER, XI_DIFF, nullptr, s->f32buf, s->r32, s->pin + 48);
        // a block of FP32 sweeps: plain (phase A) and defect-correction (inner)
        const unsigned ma = mask_of(PH_A), mi = mask_of(PH_INNER);
        const int blk = std::max(1, std::min(kResidualEvery, max_iter - total + 1));
        if (ma || mi) {
            for (int b = 0; b < blk; ++b) {
                if (ma) block_sweep(ma, b, blk, Z_ITER, false, nullptr, 0);
                if (mi) block_sweep(mi, b, blk, Z_ITER_NOB, true, s->r32, 8);
            }
            total += blk - 1;
        }
        cudaError_t ce = cudaStreamSynchronize(st);
        if (ce == cudaSuccess && (me || mo)) ce = cudaStreamSynchronize(st64);
        if (ce != cudaSuccess) {
            set_error("CUDA error: %s", cudaGetErrorString(ce));
            err = HMG_CUDA_ERROR;
            break;
        }
        if (tr) tr->collect();
        // equilibrium tests (step 1 in FP64)
        for (int sl = 0; sl < g.nslots; ++sl) {
            if (!((me >> sl) & 1u)) continue;
            double nrm = 0.0;
            for (int c = 0; c < 3; ++c) {
                flux[sl][c] = h[16 + sl * 3 + c] / (double)g.N3;
                nrm += flux[sl][c] * flux[sl][c];
            }
            eps_eq[sl] = std::sqrt(h[32 + sl]) / std::sqrt(nrm);
            if (eps_eq[sl] < tol) {
                status[sl] = HMG_OK;
                state[sl] = PH_DONE;
            } else {
                // the test ran on the iterate whose FP64 sweep gave eps_comp: aim the next
                // correction solve at the ratio it measured
                if (eps_comp[sl] > 0.0) qeq[sl] = std::max(qeq[sl], eps_eq[sl] / eps_comp[sl]);
                state[sl] = PH_INNER;
                best[sl] = INFINITY;
                since_best[sl] = 0;
                ++rounds;
            }
        }
        // FP64 correction sweeps
        for (int sl = 0; sl < g.nslots; ++sl) {
            if (!((mo >> sl) & 1u)) continue;
            ++iters[sl];
            ++it64[sl];
            eps_comp[sl] = eps_from_sum(h[48 + sl], sl);
            outer_eps[sl] = eps_comp[sl];
            if (!std::isfinite(eps_comp[sl])) {
                status[sl] = HMG_DIVERGED;
                state[sl] = PH_DONE;
            } else if (eps_comp[sl] < tol) {
                state[sl] = PH_EQ;
            } else {
                state[sl] = PH_INNER;
                best[sl] = INFINITY;
                since_best[sl] = 0;
                ++rounds;
            }
        }
        // FP32 blocks
        unsigned to_outer_a = 0, to_outer_i = 0;
        for (int sl = 0; sl < g.nslots; ++sl) {
            const bool a = (ma >> sl) & 1u, in = (mi >> sl) & 1u;
            if (!a && !in) continue;
            iters[sl] += blk;
            eps32[sl] = eps_from_sum(a ? h[sl] : h[8 + sl], sl);
            if (!std::isfinite(eps32[sl])) {
                status[sl] = HMG_DIVERGED;
                state[sl] = PH_DONE;
                continue;
            }
            if (eps32[sl] < best[sl] * improve) {
                best[sl] = eps32[sl];
                since_best[sl] = 0;
            } else {
                since_best[sl] += blk;
            }
            if (a) {
                eps_comp[sl] = eps32[sl];
                if (eps32[sl] < thetaA || since_best[sl] >= stall) to_outer_a |= 1u << sl;
            } else if (eps32[sl] < std::max(eta * outer_eps[sl], inner_target(tol, qeq[sl])) || since_best[sl] >= stall) {
                to_outer_i |= 1u << sl;
            }
        }
        if (to_outer_a) HMG_TRACED(HMG_K_OTHER, 0.0, launch_widen(g, to_outer_a, s->f32buf, s->tau64, st));
        if (to_outer_i) HMG_TRACED(HMG_K_OTHER, 0.0, launch_axpy(g, to_outer_i, s->f32buf, s->tau64, st));
        for (int sl = 0; sl < g.nslots; ++sl)
            if (((to_outer_a | to_outer_i) >> sl) & 1u) state[sl] = PH_OUTER;
    }
    cudaEventDestroy(ready);
    if (err != HMG_OK) return err;
    if ((g.xpers || g.zpers) && fast_take_wait_failure()) {
        set_error("a persistent kernel gave up waiting for its bulk copies; results are invalid");
        return HMG_CUDA_ERROR;
    }
    unsigned left = 0;
    for (int sl = 0; sl < g.nslots; ++sl)
        if (status[sl] == HMG_NOT_CONVERGED) {
            if (state[sl] == PH_A) HMG_TRACED(HMG_K_OTHER, 0.0, launch_widen(g, 1u << sl, s->f32buf, s->tau64, st));
            if (state[sl] == PH_INNER) HMG_TRACED(HMG_K_OTHER, 0.0, launch_axpy(g, 1u << sl, s->f32buf, s->tau64, st));
            left |= 1u << sl;
        }
    if (left && !check_eq<double>(left, s->tau64, s->spec64, eps_eq, flux)) return HMG_CUDA_ERROR;
    return finish(status, iters, it64, eps_comp, eps_eq, flux, rounds, info, K);
}

hmg_status Solver::finish(const int status[3], const int iters[3], const int it64[3], const double eps_comp[3],
                          const double eps_eq[3], const double flux[3][3], int rounds, hmg_info* info,
                          double K[9]) {
    for (int j = 0; j < 3; ++j)
        for (int i = 0; i < 3; ++i) K[3 * i + j] = j < g.nslots ? flux[j][i] : 0.0;
    if (info) {
        for (int j = 0; j < 3; ++j) {
            info->iters[j] = iters[j];
            info->iters_fp64[j] = it64[j];
            info->eps_comp[j] = eps_comp[j];
            info->eps_eq[j] = eps_eq[j];
            info->status[j] = status[j];
        }
        info->fp64_rounds = rounds;
    }
    for (int j = 0; j < g.nslots; ++j)
        if (status[j] != HMG_OK) return (hmg_status)status[j];
    return HMG_OK;
}

template void Solver::sweep<float>(unsigned, float*, void*, int, int, const float*, float*, float*, double*, const StopRule&);
template void Solver::sweep<double>(unsigned, double*, void*, int, int, const float*, float*, float*, double*, const StopRule&);
template void Solver::sweeps<float>(unsigned, float*, void*, int, double*, int, const StopRule&);
template void Solver::sweeps<double>(unsigned, double*, void*, int, double*, int, const StopRule&);
template bool Solver::check_eq<float>(unsigned, const float*, void*, double*, double (*)[3]);
template bool Solver::check_eq<double>(unsigned, const double*, void*, double*, double (*)[3]);

}  // namespace hmg
