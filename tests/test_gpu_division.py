"""The field from the polarization variable, e = tau / (k + k0), against the division itself: a
call of no sweeps takes e to tau = (k + k0) e and back, so its result is the IEEE quotient of
the rounded product, bit for bit, at every size of the operands."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1504_07499_gb300 import hmg

N = 16


def _values(rng):
    """Magnitudes from the subnormals up, signed zeros, infinities, NaN."""
    e = rng.uniform(1.0, 2.0, (3, N, N, N)) * rng.choice([-1.0, 1.0], (3, N, N, N))
    e = np.ldexp(e, rng.integers(-1076, 1020, e.shape) * (rng.random(e.shape) < 0.5))
    flat = e.reshape(-1)
    flat[rng.integers(0, flat.size, 60)] = np.repeat([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324], 10)
    return e


@pytest.mark.parametrize("prec", [hmg.HMG_FP64, hmg.HMG_FP32_BULK])
@pytest.mark.parametrize("lo,hi", [(0.01, 100.0), (1.0, 2.0), (1e-100, 1e100)])
def test_field_is_the_ieee_quotient(prec, lo, hi):
    rng = np.random.default_rng(int(1e6 * lo) + prec)
    with hmg.Context(0) as ctx, np.errstate(all="ignore"):
        for _ in range(60):
            k = np.exp(rng.uniform(np.log(lo), np.log(hi), 3))
            ph = rng.integers(0, 3, (N, N, N)).astype(np.uint8)
            e = _values(rng)
            kp = (k + np.sqrt(k.min() * k.max()))[ph]
            tau = kp * e
            if prec == hmg.HMG_FP32_BULK:
                tau = tau.astype(np.float32).astype(np.float64)
            want = tau / kp
            hmg.hmg_em_iterate(ctx.handle, ph, N, tuple(k), (1.0, 0.0, 0.0), prec, 0, e)
            nan = np.isnan(want)
            assert np.array_equal(np.isnan(e), nan)
            assert np.array_equal(e[~nan].view(np.int64), want[~nan].view(np.int64))
