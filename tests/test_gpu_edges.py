"""Edges of the ranges that choose a kernel or a route: row tails and many spheres in the
voxelizer, placements beyond one block of spheres, sweeps in one call against sweeps call by
call, iteration caps inside a block of sweeps, transforms on the caller's own memory.

Whole numbers and placements are equal.  Sweeps taken one call at a time pass through the
gradient field between calls: a few roundings of the working precision per sweep and no
cancellation beyond the contrast, so 1e-12 (FP64) and 1e-5 (FP32) of the field.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import em as om
from paper_1504_07499_gb300 import hmg, inputs as I

K3 = (0.20, 0.25, 40.0)


@pytest.fixture(scope="module")
def ctx():
    with hmg.Context(0) as c:
        yield c


@pytest.mark.parametrize("N,n,f", [(8, 3, 0.3), (12, 600, 0.2), (54, 600, 0.25), (72, 1, 0.45), (162, 40, 0.3)])
def test_voxelize_row_tails_and_unaligned_output(ctx, N, n, f):
    sph = np.column_stack([I.rsa(N, n, I.sphere_radius(n, f)), np.full(n, I.sphere_radius(n, f))])
    sph[:, :3] = (sph[:, :3] - sph[0, :3] + (0.0, 1.0 - 2.0 ** -22, 0.5)) % 1.0   # the first one on the cell's seams
    ref = om.voxelize(sph, 0.3, N)
    buf = torch.full((N ** 3 + 2,), 77, dtype=torch.uint8, device="cuda")
    hmg.hmg_voxelize(ctx.handle, sph, 0.3, N, buf[1:])
    got = buf.cpu().numpy()
    assert got[0] == 77 and got[-1] == 77
    assert np.array_equal(got[1:-1].reshape(N, N, N), ref)


@pytest.mark.parametrize("n,f,cap", [(33, 0.40, 20000), (129, 0.40, 20000), (260, 0.38, 20000), (320, 0.33, 400000),
                                     (1024, 0.31, 400000)])
def test_placement_beyond_one_block(ctx, n, f, cap):
    r = I.sphere_radius(n, f)
    ref = I.rsa(5, n, r, max_candidates=cap)
    grown = ref is None
    if grown:
        ref = I.grow_mc(5, I.rsa(5, n, 0.85 * r, max_candidates=cap, stream=2), r)
    got, gen = hmg.hmg_rsa(ctx.handle, 5, n, r, max_candidates=cap)
    assert gen == grown
    assert np.array_equal(got[:, :3], ref)


@pytest.mark.parametrize("prec,tol,N", [(hmg.HMG_FP64, 1e-12, n) for n in (8, 36, 64, 96, 108)] +
                         [(hmg.HMG_FP32_BULK, 1e-5, n) for n in (12, 64, 96, 128, 192, 256)])
def test_sweeps_in_one_call_match_single_calls(ctx, prec, tol, N):
    ph = I.random_phase_grid(N, N)
    E = np.array([0.3, -1.0, 0.5])
    e0 = torch.from_numpy(E).cuda()[:, None, None, None].expand(3, N, N, N).contiguous()
    a, b = e0.clone(), e0.clone()
    eps_a = hmg.hmg_em_iterate(ctx.handle, ph, N, K3, E, prec, 4, a)
    eps_b = [hmg.hmg_em_iterate(ctx.handle, ph, N, K3, E, prec, 1, b)[0] for _ in range(4)]
    assert float((a - b).abs().max()) < tol * float(a.abs().max())
    assert np.allclose(eps_a, eps_b, rtol=max(tol, 1e-11) * 100)


@pytest.mark.parametrize("m", [1, 2, 3, 7, 8, 9, 10])
def test_iteration_cap_inside_a_block(ctx, m):
    N = 24
    ph = I.random_phase_grid(1, N)
    e = np.empty((3, 3, N, N, N))
    _, info, st = hmg.hmg_solve_fields(ctx.handle, ph, N, K3, 1e-13, hmg.HMG_FP64, e, max_iter=m,
                                       allow=(hmg.HMG_OK, hmg.HMG_NOT_CONVERGED))
    assert st == hmg.HMG_NOT_CONVERGED and list(info["iters"]) == [m] * 3
    for s in range(3):
        E = np.eye(3)[s]
        ref = np.broadcast_to(E[:, None, None, None], (3, N, N, N)).copy()
        hmg.hmg_em_iterate(ctx.handle, ph, N, K3, E, hmg.HMG_FP64, m, ref)
        assert np.abs(e[s] - ref).max() < 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("prec", [hmg.HMG_FP64, hmg.HMG_FP32_BULK])
@pytest.mark.parametrize("N,count", [(24, 1), (36, 4), (64, 2), (96, 3)])
def test_transforms_on_device_memory_equal_host_memory(ctx, N, count, prec):
    x = np.random.default_rng(N).standard_normal((count, N, N, N))
    X, y = np.empty_like(x), np.empty_like(x)
    hmg.hmg_fft_forward(ctx.handle, N, count, prec, x, X)
    hmg.hmg_fft_inverse(ctx.handle, N, count, prec, X, y)
    for shift, inplace in ((0, False), (1, False), (0, True), (1, True)):   # 8 bytes off alignment; in place
        src = torch.empty(x.size + shift, dtype=torch.float64, device="cuda")[shift:]
        dst = src if inplace else torch.empty(x.size + shift, dtype=torch.float64, device="cuda")[shift:]
        src.copy_(torch.from_numpy(x).flatten())
        torch.cuda.synchronize()
        hmg.hmg_fft_forward(ctx.handle, N, count, prec, src, dst)
        assert np.array_equal(dst.cpu().numpy().reshape(x.shape), X)
        hmg.hmg_fft_inverse(ctx.handle, N, count, prec, dst, src)
        assert np.array_equal(src.cpu().numpy().reshape(x.shape), y)
