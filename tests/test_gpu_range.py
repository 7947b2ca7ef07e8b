"""FP64 transforms and sweeps at the lower end of the FP64 range: a power of two in front of a field
changes only exponents, down to the rounding of subnormal results.

Two roundings to subnormals (2^-1074 apart) of values that agree to 2^-52 differ by at most one unit.
Fields of subnormals only (one unit is 2^-34 of them) come back as accurately as FP64 operations
would give them: one unit per value in each of at most 24 radix-2 stages, 2^-29 of the norm.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1504_07499_gb300 import hmg


@pytest.fixture(scope="module")
def ctx():
    with hmg.Context(0) as c:
        yield c


def _noise(N):
    return torch.randn(N, N, N, dtype=torch.float64, device="cuda",
                       generator=torch.Generator(device="cuda").manual_seed(N))


def _up(x, p):     # exact for these values
    return x * 2.0 ** (p // 2) * 2.0 ** (p - p // 2)


def _same(got, want, p):
    d = _up(got - want, 1074)
    if p < 1040:
        assert float(d.abs().max()) <= 1.0
    else:
        assert float(d.norm()) <= 2.0 ** -29 * float(_up(want, 1074).norm())
    assert got.any()


@pytest.mark.parametrize("N", [8, 18, 32, 96, 128, 216])
@pytest.mark.parametrize("p", [1000, 1020, 1040])   # normal, partly subnormal, subnormal input
def test_transforms_of_tiny_fields(ctx, N, p):
    x = (_noise(N) * 2.0 ** -1000 * 2.0 ** -(p - 1000))[None]   # rounded to multiples of 2^-1074
    big = _up(x, 1060)
    X, Xbig, y, ybig = (torch.empty_like(x) for _ in range(4))
    hmg.hmg_fft_forward(ctx.handle, N, 1, hmg.HMG_FP64, x, X)
    hmg.hmg_fft_forward(ctx.handle, N, 1, hmg.HMG_FP64, big, Xbig)
    want = Xbig * 2.0 ** -1000 * 2.0 ** -60
    _same(X, want, p)
    # inverse of a spectrum with subnormal values: the noise again, packed
    hmg.hmg_fft_inverse(ctx.handle, N, 1, hmg.HMG_FP64, x, y)
    hmg.hmg_fft_inverse(ctx.handle, N, 1, hmg.HMG_FP64, big, ybig)
    want = ybig * 2.0 ** -1000 * 2.0 ** -60
    _same(y, want, p)


@pytest.mark.parametrize("N", [8, 18, 32, 96, 128, 216])
@pytest.mark.parametrize("sweeps", [1, 3])
def test_sweeps_of_tiny_polarizations(ctx, N, sweeps):
    # Conductivities times 2^-500 and fields times 2^-510: tau = (k + k0) e is 2^-1010 of what it
    # was, so it rounds to 2^-64 of its size at most; e stays normal and may differ in its last bits.
    ph = torch.randint(0, 3, (N, N, N), device="cuda", generator=torch.Generator(device="cuda").manual_seed(N)).to(torch.uint8)
    e = torch.stack([0.3 * _noise(N) + m for m in (0.3, -1.0, 0.5)])
    E, k = np.array([0.3, -1.0, 0.5]), np.array([0.2, 0.25, 40.0])
    big, small = e.clone(), e * 2.0 ** -510
    hmg.hmg_em_iterate(ctx.handle, ph, N, k, E, hmg.HMG_FP64, sweeps, big)
    hmg.hmg_em_iterate(ctx.handle, ph, N, k * 2.0 ** -500, E * 2.0 ** -510, hmg.HMG_FP64, sweeps, small)
    assert float((small * 2.0 ** 510 - big).abs().max()) <= 2.0 ** -50 * float(big.abs().max())
