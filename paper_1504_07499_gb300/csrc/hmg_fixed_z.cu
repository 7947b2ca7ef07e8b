// FP64 z pass of a sweep or an equilibrium test in block fixed point, and its table of
// projector reciprocals.
#include "hmg_fixed_kernels.cuh"

namespace hmg {

namespace {
// rcp[n2] = round(2^60 4^b / n2), b = proj_bits(n2): in [2^60, 2^62]
__global__ void k_rcp_table(long long* rcp, int count) {
    const int n2 = blockIdx.x * blockDim.x + threadIdx.x;
    if (n2 >= count) return;
    if (n2 == 0) {
        rcp[0] = 0;
        return;
    }
    const int s = 2 * fx::proj_bits(n2) - 2;
    const unsigned long long n = (unsigned long long)n2, one = 1ull << 62, q = one / n, r = one % n;
    rcp[n2] = (long long)((q << s) + ((r << s) + n / 2) / n);
}
}  // namespace

void fx_rcp_table(long long* rcp, int N) {
    const int count = fx_rcp_count(N);
    k_rcp_table<<<(count + 255) / 256, 256>>>(rcp, count);
}

int fx_z_ctas(const GridDesc& g) {
    switch (g.N) {
#define X(N_) \
    case N_: return N_ * (N_ / 2 / fx::ZShape<N_>::NP);
        HMG_ALL_SIZES(X)
#undef X
        default: return 0;
    }
}

void fx_z(const GridDesc& g, int mode, unsigned mask, void* spec, double* partial, cudaStream_t st) {
    fx::c64* sp = reinterpret_cast<fx::c64*>(spec);
    const dim3 grid(fx_z_ctas(g), g.nslots);
    switch (g.N) {
#define X(N_)                                                                                             \
    case N_:                                                                                              \
        fx::launch(fx::k_fxx_z<N_>, grid, fx::ZShape<N_>::T, fx::ZShape<N_>::smem, st, g, mask, mode, sp, partial); \
        break;
        HMG_ALL_SIZES(X)
#undef X
    }
}

}  // namespace hmg
