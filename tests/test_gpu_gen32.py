"""FP32 kernels of the grid sizes outside hmg_fast.cu: transforms and sweeps at every size, and
chained against unchained sweeps.

Tolerances as in test_gpu_parity: FP32 transforms 2e-6 of the largest coefficient, FP32
sweeps 1e-5 relative; chaining changes no float operation, so its results are equal bit for bit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import em as om
from paper_1504_07499_gb300 import hmg, inputs as I

SIZES = [8, 12, 16, 18, 24, 32, 36, 48, 54, 72, 108, 144, 162, 216, 288, 324, 384, 432, 486]
K3 = I.K_PHASES


@pytest.fixture(scope="module")
def ctx():
    with hmg.Context(0) as c:
        yield c


@pytest.mark.parametrize("N", SIZES)
def test_transforms(ctx, N):
    g = torch.Generator(device="cuda").manual_seed(N)
    x = torch.randn(2, N, N, N, dtype=torch.float64, device="cuda", generator=g)
    X, y = torch.empty_like(x), torch.empty_like(x)
    torch.cuda.synchronize()
    hmg.hmg_fft_forward(ctx.handle, N, 2, hmg.HMG_FP32_BULK, x, X)
    hmg.hmg_fft_inverse(ctx.handle, N, 2, hmg.HMG_FP32_BULK, X, y)
    for i in range(2):
        h = torch.fft.rfftn(x[i])
        ref = h[..., :N // 2].clone()
        ref[..., 0] += 1j * h[..., N // 2]
        got = torch.view_as_complex(X[i].reshape(N, N, N // 2, 2))
        assert float((got - ref).abs().max()) < 2e-6 * float(ref.abs().max())
        assert float((y[i] / N ** 3 - x[i]).abs().max()) < 2e-5 * float(x[i].abs().max())


@pytest.mark.parametrize("N", [n for n in SIZES if n <= 54])
def test_sweeps_match_oracle(ctx, N):
    ph = I.random_phase_grid(N, N)
    E = np.array([0.3, -1.0, 0.5])
    e0 = E[:, None, None, None] + 0.3 * np.random.default_rng(N).standard_normal((3, N, N, N))
    ref = om.em_solve(ph, K3, E, tol=0.0, max_iter=2, record=True, e0=e0)
    e = e0.copy()
    eps = hmg.hmg_em_iterate(ctx.handle, ph, N, K3, E, hmg.HMG_FP32_BULK, 2, e)
    assert np.abs(e - ref.e).max() < 1e-5 * np.abs(ref.e).max()
    assert np.allclose(eps, ref.eps_comp_hist, rtol=1e-4)


@pytest.mark.parametrize("N", [8, 12, 18, 36, 54, 108, 162, 216])
def test_chained_sweeps_are_bit_identical(ctx, N):
    ph = I.random_phase_grid(N, N)
    k = (0.20, 0.25, 2.0)
    out = []
    for variant in (0, 4):   # chained, unchained
        hmg.hmg_set_variant(ctx.handle, N, variant)
        e = torch.empty(3, 3, N, N, N, dtype=torch.float64, device="cuda")
        K, info, _ = hmg.hmg_solve_fields(ctx.handle, ph, N, k, 1e-8, hmg.HMG_FP32_BULK, e)
        Kb, _, _ = hmg.hmg_solve_batch(ctx.handle, [ph, ph], [N, N], [k, k], 1e-8, hmg.HMG_FP32_BULK)
        out.append((K, e, info["iters"], Kb))
    hmg.hmg_set_variant(ctx.handle, N, -1)
    assert (out[0][0] == out[1][0]).all() and torch.equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2] and (out[0][3] == out[1][3]).all()
