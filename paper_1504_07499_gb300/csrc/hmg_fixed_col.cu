// FP64 column passes in block fixed point (y passes; z passes of a plain transform).
#include "hmg_fixed_kernels.cuh"

namespace hmg {

namespace {
template <bool PLAIN>
void col(const GridDesc& g, unsigned mask, const void* src, void* spec, const fx::ColArgs& a, cudaStream_t st) {
    const fx::c64* in = reinterpret_cast<const fx::c64*>(src);
    fx::c64* sp = reinterpret_cast<fx::c64*>(spec);
    switch (g.N) {
#define X(N_)                                                                                          \
    case N_:                                                                                           \
        fx::launch(fx::k_fxx_col<N_, PLAIN>, dim3(g.comps * N_ * (N_ / 2 / fx::ColShape<N_>::NP), g.nslots), \
                   fx::ColShape<N_>::T, fx::ColShape<N_>::smem, st, g, mask, in, sp, a);                 \
        break;
        HMG_ALL_SIZES(X)
#undef X
    }
}
}  // namespace

void fx_y(const GridDesc& g, bool forward, unsigned mask, void* spec, cudaStream_t st) {
    col<false>(g, mask, spec, spec, fx::ColArgs{forward ? 0 : 1, g.expA, g.expB}, st);
}

void fx_z_plain(const GridDesc& g, bool forward, unsigned mask, const void* src, void* spec, cudaStream_t st) {
    col<true>(g, mask, src, spec, fx::ColArgs{forward ? 0 : 1, g.expB, g.expA}, st);
}

}  // namespace hmg
