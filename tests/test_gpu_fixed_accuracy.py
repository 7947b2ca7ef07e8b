"""FP64 forward transforms against extended precision: fields that are exact products of integer
vectors, whose transform is the product of three 1D sums in long double (64 bits of fraction or more).

Bounds: a pass errs by about two quanta per component, a quantum is 2^-58 of a pencil's largest
value.  That is at most 5 times the pencil's rms in zero-mean noise and sqrt(72) times in the spectra
of a field with a mean: 2^-54.7 and 2^-53.9 of the norm per pass, sqrt(3) times that in three, and
the rounding of the result to FP64 (2^-54): below 2^-53 and 1.5 2^-53.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1504_07499_gb300 import hmg

SIZES = [n for n in sorted(2 ** a * 3 ** b for a in range(1, 7) for b in range(5)) if 8 <= n <= 72]


def _dft(v):
    """Long-double DFT of an integer vector, angles reduced in integers."""
    N = len(v)
    q = np.outer(np.arange(N), np.arange(N)) % N
    ang = q.astype(np.longdouble) * (8 * np.arctan(np.longdouble(1)) / N)
    x = v.astype(np.longdouble)
    re, im = (np.cos(ang) * x).sum(axis=1), (-np.sin(ang) * x).sum(axis=1)
    return re + 1j * im


@pytest.mark.parametrize("mean", [False, True])
@pytest.mark.parametrize("N", SIZES)
def test_forward_against_long_double(N, mean):
    rng = np.random.default_rng(N)
    a, b, c = (rng.integers(0 if mean else -40000, 40000, N) for _ in range(3))   # products below 2^53
    x = c[:, None, None].astype(np.float64) * b[None, :, None] * a[None, None, :]
    X = np.empty(2 * x.size // 2)
    with hmg.Context(0) as ctx:
        hmg.hmg_fft_forward(ctx.handle, N, 1, hmg.HMG_FP64, x, X)
    A, B, C = _dft(a), _dft(b), _dft(c)
    ref = C[:, None, None] * B[None, :, None] * A[None, None, :N // 2]
    ref[..., 0] += 1j * (C[:, None] * B[None, :] * A[N // 2])
    got = X.reshape(N, N, N // 2, 2)
    d = got[..., 0].astype(np.longdouble) + 1j * got[..., 1].astype(np.longdouble) - ref
    err = np.sqrt((abs(d) ** 2).sum() / (abs(ref) ** 2).sum())
    print(f"{N} {'mean' if mean else 'noise'} {float(err):.2e}")
    assert err <= (1.5 if mean else 1.0) * 2.0 ** -53
