// FP64 x passes in block fixed point: launchers over the grid sizes.
#include "hmg_fixed_kernels.cuh"

namespace hmg {

int fx_x_ctas(const GridDesc& g) {
    switch (g.N) {
#define X(N_) \
    case N_: return (int)(g.comps * g.NN / fx::x_rows<N_ / 2>());
        HMG_ALL_SIZES(X)
#undef X
        default: return 0;
    }
}

void fx_x_forward(const GridDesc& g, int mode, unsigned mask, const double* tau, void* spec, double* partial,
                  cudaStream_t st) {
    fx::c64* sp = reinterpret_cast<fx::c64*>(spec);
    const dim3 grid(fx_x_ctas(g), g.nslots);
    switch (g.N) {
#define X(N_)                                                                                            \
    case N_:                                                                                             \
        fx::launch(fx::k_fxx_forward<N_ / 2>, grid, fx::XShape<N_ / 2>::T, fx::XShape<N_ / 2>::smem, st, g, mask, \
                   mode, tau, sp, partial);                                                              \
        break;
        HMG_ALL_SIZES(X)
#undef X
    }
}

void fx_x_inverse(const GridDesc& g, int mode, unsigned mask, const void* spec, double* tau, float* d32, float* r32,
                  double* partial, cudaStream_t st) {
    const fx::c64* sp = reinterpret_cast<const fx::c64*>(spec);
    const dim3 grid(fx_x_ctas(g), g.nslots);
    switch (g.N) {
#define X(N_)                                                                                            \
    case N_:                                                                                             \
        fx::launch(fx::k_fxx_inverse<N_ / 2>, grid, fx::XShape<N_ / 2>::T, fx::XShape<N_ / 2>::smem, st, g, mask, \
                   mode, sp, tau, d32, r32, partial);                                                    \
        break;
        HMG_ALL_SIZES(X)
#undef X
    }
}

void fx_x_round(const GridDesc& g, unsigned mask, void* spec, double* tau, double* partial, cudaStream_t st) {
    fx::c64* sp = reinterpret_cast<fx::c64*>(spec);
    const dim3 grid(fx_x_ctas(g), g.nslots);
    switch (g.N) {
#define X(N_)                                                                                            \
    case N_:                                                                                             \
        fx::launch(fx::k_fxx_round<N_ / 2>, grid, fx::XShape<N_ / 2>::T, fx::XShape<N_ / 2>::smem, st, g, mask, \
                   sp, tau, partial);                                                                    \
        break;
        HMG_ALL_SIZES(X)
#undef X
    }
}

}  // namespace hmg
