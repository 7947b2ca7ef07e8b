"""FP32 sums of the x passes that take two rows at once: each row is summed by itself before FP64,
so a row of large values does not swallow its neighbour (mean flux of rows +A, b, -A, b)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1504_07499_gb300 import hmg


@pytest.mark.parametrize("N", [64, 96, 128, 192, 256])
def test_mean_flux_of_unlike_rows(N):
    # k = 1: the flux is e.  Every value and every sum of up to 48 equal ones is a float, and
    # FP64 adds the rows' sums exactly
    e = torch.ones(3, N, N, N, dtype=torch.float64, device="cuda")
    e[:, :, 0::4] = 2.0 ** 30
    e[:, :, 2::4] = -2.0 ** 30
    torch.cuda.synchronize()
    with hmg.Context(0) as ctx:
        _, flux = hmg.hmg_equilibrium(ctx.handle, np.zeros((N, N, N), np.uint8), N, (1.0, 1.0, 1.0),
                                      hmg.HMG_FP32_BULK, e)
    assert list(flux) == [0.5] * 3
