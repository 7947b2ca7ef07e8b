"""Paths of a solve and of the placement that the other tests do not reach: a residual that is not a number
under the device flags of a plain FP64 solve, fields into device memory off the 16-byte grid, and a
candidate filter with thousands of survivors."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1504_07499_gb300 import hmg, inputs as I


@pytest.fixture(scope="module")
def ctx():
    with hmg.Context(0) as c:
        yield c


@pytest.mark.parametrize("N", [8, 32, 96])
def test_fp64_residual_that_is_not_a_number_ends_the_solve(ctx, N):
    # k0 = sqrt(min k max k) overflows: every polarization factor is NaN from the first sweep on
    ph = I.random_phase_grid(1, N)
    K, info, st = hmg.hmg_solve(ctx.handle, ph, N, (1e200, 2e200, 3e200), 1e-8, hmg.HMG_FP64, 50,
                                allow=(hmg.HMG_DIVERGED,))
    assert st == hmg.HMG_DIVERGED
    assert list(info["status"])[:3] == [hmg.STATUS_NAMES[hmg.HMG_DIVERGED]] * 3
    assert list(info["iters"])[:3] == [1, 1, 1]
    K, info, st = hmg.hmg_solve(ctx.handle, ph, N, (0.2, 0.25, 2.0), 1e-8, hmg.HMG_FP64)   # and the next one runs
    assert st == hmg.HMG_OK and np.isfinite(K).all()


@pytest.mark.parametrize("prec", [hmg.HMG_FP64, hmg.HMG_FP32_BULK])
def test_fields_into_unaligned_device_memory(ctx, prec):
    N, k = 24, (0.2, 0.25, 2.0)
    ph = torch.from_numpy(I.random_phase_grid(1, N)).cuda()
    buf = torch.zeros(9 * N ** 3 + 3, dtype=torch.float64, device="cuda")
    good = torch.zeros(9 * N ** 3, dtype=torch.float64, device="cuda")
    off = buf[1:1 + 9 * N ** 3]
    assert off.data_ptr() % 16 == 8 and good.data_ptr() % 16 == 0
    Ka, _, _ = hmg.hmg_solve_fields(ctx.handle, ph, N, k, 1e-8, prec, good)
    Kb, _, _ = hmg.hmg_solve_fields(ctx.handle, ph, N, k, 1e-8, prec, off)
    torch.cuda.synchronize()
    assert np.array_equal(Ka, Kb) and torch.equal(off, good) and good.any()
    assert float(buf[0]) == 0.0 and not buf[1 + 9 * N ** 3:].any()


@pytest.mark.parametrize("seed,f", [(21, 0.24), (22, 0.28)])
def test_filtered_candidates_of_1024_spheres(ctx, seed, f):
    # about 3200 and 2400 survivors of the first filtered chunk
    r = I.sphere_radius(1024, f)
    got, gen = hmg.hmg_rsa(ctx.handle, seed, 1024, r)
    assert gen == 0 and np.array_equal(got[:, :3], I.rsa(seed, 1024, r))
