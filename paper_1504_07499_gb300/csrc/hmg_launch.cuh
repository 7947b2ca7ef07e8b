// Kernel launches that overlap with the end of the kernel before (programmatic dependent
// launch): the grid's CTAs are scheduled while the last CTAs of the predecessor in the stream
// still run, and wait in grid_begin() until it has finished and its writes are visible.  This
// hides launch latency and prologues between the short dependent kernels of a sweep.
// Only for spectra that fit in L2 (small_grid): FP32-bulk sweeps of three gradients went 38.5 -> 28
// us at 64^3, 78 -> 66 at 96^3 and 131 -> 118 at 128^3, but 510 -> 540 at 192^3 and 978 -> 1150 at
// 256^3 -- the waiting CTAs bring nothing to kernels of 100 us and more, and a persistent
// kernel that needs most of an SM's shared memory cannot fill the SM while the kernel before
// still holds it with a smaller split between cache and shared memory.
// Every kernel launched this way calls grid_begin() in every thread before it touches memory
// that another kernel writes (and before any early exit, so that a kernel never finishes
// ahead of its predecessors); tables that no kernel writes may be read earlier.  Its lifetime begins
// while the kernel before still writes, and the read-only path (__ldg, or a restrict pointer that
// the kernel only reads) is defined only for data that nothing writes in that time: what another
// kernel writes is read through plain pointers, only the tables by __ldg.
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "hmg_internal.h"

namespace hmg {

#ifdef __CUDACC__
__device__ __forceinline__ void grid_begin() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the next kernel may be scheduled
    asm volatile("griddepcontrol.wait;" ::: "memory");                // the one before has finished
}

// The launch's spectrum (word: bytes per real) is at most 96 MB of the 129 MB L2.
inline bool small_grid(const GridDesc& g, size_t word) { return g.nslots * 3 * (size_t)g.N3 * word <= (96u << 20); }

// overlap: as above, else an ordinary launch
template <class... P, class... A>
void launch_kernel(bool overlap, void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = overlap ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kern, P(std::forward<A>(args))...);
}
#endif

}  // namespace hmg
