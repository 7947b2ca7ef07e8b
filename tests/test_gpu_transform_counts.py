"""FP32 transforms of one, two and more fields at the sizes with their own column kernels: every field
alone has the bits it has among others, and both directions agree with torch in FP64.

FP32: three passes each way of a few roundings (2^-24) per stage, 2^-20 of the norm.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1504_07499_gb300 import hmg


@pytest.fixture(scope="module")
def ctx():
    with hmg.Context(0) as c:
        yield c


def _packed(X, N):   # rfftn -> N/2 complex per row, kx = 0 packing X(0) + i X(N/2)
    p = X[..., :N // 2].clone()
    p[..., 0] += 1j * X[..., N // 2]
    return p


@pytest.mark.parametrize("N", [64, 96, 128, 192, 256, 512])
def test_counts(ctx, N):
    x = torch.randn(4 if N < 512 else 2, N, N, N, dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(N)) + 0.25
    n = len(x)
    one, back = torch.empty_like(x), torch.empty_like(x)
    for c in range(n):
        hmg.hmg_fft_forward(ctx.handle, N, 1, hmg.HMG_FP32_BULK, x[c], one[c])
        ref = _packed(torch.fft.rfftn(x[c]), N)
        got = torch.view_as_complex(one[c].view(N, N, N // 2, 2))
        assert float((got - ref).norm()) <= 2.0 ** -20 * float(ref.norm())
        hmg.hmg_fft_inverse(ctx.handle, N, 1, hmg.HMG_FP32_BULK, one[c], back[c])
        assert float((back[c] / N ** 3 - x[c]).norm()) <= 2.0 ** -19 * float(x[c].norm())
    for count in range(2, n + 1):
        X, y = torch.empty_like(x[:count]), torch.empty_like(x[:count])
        hmg.hmg_fft_forward(ctx.handle, N, count, hmg.HMG_FP32_BULK, x[:count], X)
        hmg.hmg_fft_inverse(ctx.handle, N, count, hmg.HMG_FP32_BULK, X, y)
        assert torch.equal(X, one[:count]) and torch.equal(y, back[:count])
