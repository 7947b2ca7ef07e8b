"""Host allocations of a solve that fail or repeat: the library's own objects are linked once more
with the CUDA runtime's pinned-memory calls wrapped (a counter and an error code on request; no
GPU fault is caused)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1504_07499_gb300 import build, hmg, inputs as I

WRAP = r"""
#include <stddef.h>
int wrap_fail, wrap_made, wrap_freed;
int __real_cudaHostAlloc(void** p, size_t n, unsigned flags);   /* what C++'s cudaMallocHost calls */
int __real_cudaFreeHost(void* p);
int __wrap_cudaHostAlloc(void** p, size_t n, unsigned flags) {
    if (wrap_fail) return 2;   /* cudaErrorMemoryAllocation */
    ++wrap_made;
    return __real_cudaHostAlloc(p, n, flags);
}
int __wrap_cudaFreeHost(void* p) {
    ++wrap_freed;
    return __real_cudaFreeHost(p);
}
"""


@pytest.fixture(scope="module")
def wrapped(tmp_path_factory):
    """The library with wrapped allocations: (path, its counters)."""
    build.build()
    objs = [os.path.join(build.BUILD, os.path.splitext(s)[0] + ".o") for s in build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    d = tmp_path_factory.mktemp("wrap")
    (d / "wrap.c").write_text(WRAP)
    subprocess.run(["gcc", "-c", "-fPIC", str(d / "wrap.c"), "-o", str(d / "wrap.o")], check=True)
    so = str(d / "libhmg_wrapped.so")
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-o", so, *objs, str(d / "wrap.o"), "-lcudart",
                    "-Xlinker", "--wrap=cudaHostAlloc", "-Xlinker", "--wrap=cudaFreeHost"], check=True)
    return so


@pytest.fixture
def lib(wrapped, monkeypatch):
    monkeypatch.setattr(hmg, "LIB_PATH", wrapped)
    monkeypatch.setattr(hmg, "_lib", None)
    L = hmg.lib()
    ctypes.c_int.in_dll(L, "wrap_fail").value = 0
    return lambda name: ctypes.c_int.in_dll(L, name)


@pytest.mark.parametrize("prec", [hmg.HMG_FP64, hmg.HMG_FP32_BULK])
def test_no_pinned_memory_is_an_error_and_writes_nothing(lib, prec):
    N = 16
    ph = I.random_phase_grid(1, N)
    e = np.full((3, 3, N, N, N), 7.0)
    K, info = np.full(9, 7.0), hmg.hmg_info()
    info.status[0] = 7
    with hmg.Context(0) as ctx:
        lib("wrap_fail").value = 1
        st = hmg.lib().hmg_solve_fields(ctx.handle, ph.ctypes.data, N, 0.2, 0.25, 2.0, 1e-8, prec, 0, hmg._dbuf(K),
                                        ctypes.byref(info), e.ctypes.data)
        lib("wrap_fail").value = 0
        assert st == hmg.HMG_OUT_OF_MEMORY
        assert (e == 7.0).all() and (K == 7.0).all() and info.status[0] == 7
        ok, _, _ = hmg.hmg_solve_fields(ctx.handle, ph, N, (0.2, 0.25, 2.0), 1e-8, prec, e)   # and the context goes on
    assert np.isfinite(ok).all() and not (e == 7.0).any()


def test_pinned_memory_is_made_once_per_context(lib):
    made, freed = lib("wrap_made"), lib("wrap_freed")
    m0, f0 = made.value, freed.value
    with hmg.Context(0) as ctx:
        for N in (16, 24, 16, 32):
            for prec in (hmg.HMG_FP64, hmg.HMG_FP32_BULK):
                hmg.hmg_solve(ctx.handle, I.random_phase_grid(1, N), N, (0.2, 0.25, 2.0), 1e-6, prec)
        assert (made.value - m0, freed.value - f0) == (1, 0)
    assert (made.value - m0, freed.value - f0) == (1, 1)
