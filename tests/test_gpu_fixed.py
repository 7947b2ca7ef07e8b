"""FP64 passes in block fixed point: every grid size against numpy, scaling, zeros, non-finite values."""
import numpy as np
import pytest

from paper_1504_07499_gb300 import hmg

pytestmark = pytest.mark.gpu
SIZES = sorted(2 ** a * 3 ** b for a in range(1, 10) for b in range(6) if 8 <= 2 ** a * 3 ** b <= 512)


@pytest.fixture(scope="module")
def ctx():
    with hmg.Context(0) as c:
        yield c


def _fields(N):
    """Noise, a two-phase field far from zero mean, and a smooth field."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(N)
    x = torch.randn(3, N, N, N, dtype=torch.float64, device="cuda", generator=g)
    x[1] = (x[1] > 2.0).double() * 400 + 0.2
    a = torch.arange(N, device="cuda", dtype=torch.float64) * (2 * np.pi / N)
    x[2] = torch.cos(a)[:, None, None] * torch.sin(2 * a)[None, :, None] * torch.exp(torch.cos(a)) + 3
    return x


def _round_trip(ctx, N, x):
    import torch
    X, y = torch.empty_like(x), torch.empty_like(x)
    hmg.hmg_fft_forward(ctx.handle, N, len(x), hmg.HMG_FP64, x, X)
    hmg.hmg_fft_inverse(ctx.handle, N, len(x), hmg.HMG_FP64, X, y)
    torch.cuda.synchronize()
    return X, y


@pytest.mark.parametrize("N", SIZES)
def test_round_trip_of_every_size(ctx, N):
    # six passes, each within one FP64 rounding (2^-53) of its pencils' norm: below 2^-50
    x = _fields(N)
    _, y = _round_trip(ctx, N, x)
    for c in range(3):
        assert float((y[c] / N ** 3 - x[c]).norm() / x[c].norm()) < 2.0 ** -50


@pytest.mark.parametrize("N", [n for n in SIZES if n <= 108])
def test_forward_against_numpy(ctx, N):
    # numpy's own FP64 error (a few 2^-53 at these lengths) dominates: 2^-49
    x = _fields(N)
    X, _ = _round_trip(ctx, N, x)
    for c in range(3):
        h = np.fft.rfftn(x[c].cpu().numpy())
        ref = h[..., :N // 2].copy()
        ref[..., 0] += 1j * h[..., N // 2]
        got = X[c].cpu().numpy().reshape(N, N, N // 2, 2)
        assert np.linalg.norm(got[..., 0] + 1j * got[..., 1] - ref) < 2.0 ** -49 * np.linalg.norm(ref)


@pytest.mark.parametrize("N", [12, 54, 128])
def test_scaling_zero_and_non_finite(ctx, N):
    import torch
    x = _fields(N)
    X, y = _round_trip(ctx, N, x)
    for s in (2.0 ** -600, 2.0 ** 600):   # exponents are carried apart: results scale exactly
        Xs, ys = _round_trip(ctx, N, x * s)
        assert torch.equal(Xs, X * s) and torch.equal(ys, y * s)
    x[1] = 0
    x[2, 1, 2, 3] = float("inf")
    X, y = _round_trip(ctx, N, x)
    assert not X[1].any() and not y[1].any()          # a zero grid stays zero
    assert not torch.isfinite(X[2]).any()             # every mode depends on the infinite voxel
    assert torch.isfinite(y[0]).all()
