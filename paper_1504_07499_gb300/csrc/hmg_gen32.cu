// Launchers of the FP32 passes of hmg_gen32_kernels.cuh; each returns false (launching
// nothing) for the grid sizes that hmg_fast.cu serves.
#include "hmg_gen32_kernels.cuh"

namespace hmg {

#define HMG_G32_SIZES(X)                                                                                    \
    X(8) X(12) X(16) X(18) X(24) X(32) X(36) X(48) X(54) X(72) X(108) X(144) X(162) X(216) X(288) X(324) X(384) \
    X(432) X(486)

namespace {
template <class K, class... Args>
void launch(K kern, dim3 grid, int threads, size_t smem, cudaStream_t st, const GridDesc& g, Args... args) {
    if (smem > 32 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_kernel(small_grid(g, sizeof(float)), kern, grid, threads, smem, st, g, args...);
}
}  // namespace

int gen_x_ctas(const GridDesc& g) {
    switch (g.N) {
#define X(N_) \
    case N_: return (int)(g.comps * g.NN / g32::x_rows<N_ / 2>());
        HMG_G32_SIZES(X)
#undef X
        default: return 0;
    }
}

int gen_z_ctas(const GridDesc& g) {
    switch (g.N) {
#define X(N_) \
    case N_: return N_ * (N_ / 2 / g32::ZShape<N_>::NP);
        HMG_G32_SIZES(X)
#undef X
        default: return 0;
    }
}

bool gen_x_forward(const GridDesc& g, int mode, unsigned mask, const float* tau, void* spec, double* partial,
                   cudaStream_t st) {
    const dim3 grid(gen_x_ctas(g), g.nslots);
    switch (g.N) {
#define X(N_)                                                                                              \
    case N_:                                                                                               \
        launch(mode == XF_PLAIN      ? g32::k_gx_forward<N_ / 2, XF_PLAIN>                                  \
               : mode == XF_POLARIZE ? g32::k_gx_forward<N_ / 2, XF_POLARIZE>                               \
                                     : g32::k_gx_forward<N_ / 2, XF_FLUX>,                                  \
               grid, g32::XShape<N_ / 2>::T, g32::XShape<N_ / 2>::smem, st, g, mask, tau,                   \
               reinterpret_cast<float2*>(spec), partial);                                                  \
        return true;
        HMG_G32_SIZES(X)
#undef X
        default: return false;
    }
}

bool gen_x_inverse(const GridDesc& g, int mode, unsigned mask, const void* spec, float* tau, const float* r32,
                   double* partial, cudaStream_t st) {
    const bool res = mode == XI_INPLACE_RES || mode == XI_ADD_R_RES;
    const dim3 grid(gen_x_ctas(g), g.nslots);
    switch (g.N) {
#define X(N_)                                                                                                  \
    case N_:                                                                                                   \
        launch(res ? g32::k_gx_inverse<N_ / 2, true> : g32::k_gx_inverse<N_ / 2, false>, grid,                  \
               g32::XShape<N_ / 2>::T, g32::XShape<N_ / 2>::smem, st, g, mask, mode,                            \
               reinterpret_cast<const float2*>(spec), tau, r32, partial);                                      \
        return true;
        HMG_G32_SIZES(X)
#undef X
        default: return false;
    }
}

bool gen_x_round(const GridDesc& g, bool addr, bool wtau, unsigned mask, void* spec, float* tau, const float* r32,
                 cudaStream_t st) {
    const dim3 grid(gen_x_ctas(g), g.nslots);
    switch (g.N) {
#define X(N_)                                                                                                 \
    case N_:                                                                                                  \
        launch(g32::k_gx_round<N_ / 2>, grid, g32::XShape<N_ / 2>::T, g32::XShape<N_ / 2>::smem, st, g, mask,  \
               addr ? 1 : 0, wtau ? 1 : 0, reinterpret_cast<float2*>(spec), tau, r32);                        \
        return true;
        HMG_G32_SIZES(X)
#undef X
        default: return false;
    }
}

bool gen_col(const GridDesc& g, bool zdir, bool forward, unsigned mask, void* spec, cudaStream_t st) {
    switch (g.N) {
#define X(N_)                                                                                               \
    case N_:                                                                                                \
        launch(g32::k_gcol<N_>, dim3(g.comps * N_ * (N_ / 2 / g32::ColShape<N_>::NP), g.nslots),             \
               g32::ColShape<N_>::T, g32::ColShape<N_>::smem, st, g, mask, zdir ? 1 : 0, forward ? 0 : 1,    \
               reinterpret_cast<float2*>(spec));                                                            \
        return true;
        HMG_G32_SIZES(X)
#undef X
        default: return false;
    }
}

bool gen_z(const GridDesc& g, int mode, unsigned mask, void* spec, double* partial, cudaStream_t st) {
    if (mode == Z_FWD || mode == Z_INV) return gen_col(g, true, mode == Z_FWD, mask, spec, st);
    const dim3 grid(gen_z_ctas(g), g.nslots);
    switch (g.N) {
#define X(N_)                                                                                             \
    case N_:                                                                                              \
        launch(g32::k_gz<N_>, grid, g32::ZShape<N_>::T, g32::ZShape<N_>::smem, st, g, mask, mode,          \
               reinterpret_cast<float2*>(spec), partial);                                                 \
        return true;
        HMG_G32_SIZES(X)
#undef X
        default: return false;
    }
}

}  // namespace hmg
