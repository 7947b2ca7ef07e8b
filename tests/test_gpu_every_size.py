"""Every grid size against plain FP64 torch: two sweeps, the equilibrium test and the FP64 forward
transform (the kernels have their sizes, plans and shifts fixed at compile time).

Bounds: an FP64 pass errs by at most 2^-50 of its grid's norm (test_gpu_fixed), a sweep is six of
them, torch's own transforms err by a few 2^-53 per stage, so two sweeps stay within 2^-45 of the
field's norm and the residuals and norms, which do not cancel here, within 2^-40.  FP32: 1e-5 of the
largest value and 1e-4, as in test_gpu_gen32.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1504_07499_gb300 import hmg

SIZES = sorted(2 ** a * 3 ** b for a in range(1, 10) for b in range(6) if 8 <= 2 ** a * 3 ** b <= 512)
K3 = (0.20, 0.25, 40.0)
E0 = np.array([0.3, -1.0, 0.5])


@pytest.fixture(scope="module")
def ctx():
    with hmg.Context(0) as c:
        yield c


def _inputs(N):
    g = torch.Generator(device="cuda").manual_seed(N)
    ph = torch.randint(0, 3, (N, N, N), device="cuda", generator=g).to(torch.uint8)
    e = torch.empty(3, N, N, N, dtype=torch.float64, device="cuda").normal_(generator=g)
    e *= 0.3
    for c in range(3):
        e[c] += E0[c]
    return ph, e


class Modes:
    """Signed modes of the half spectrum; Nyquist components count only where alone."""

    def __init__(self, N):
        m = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64).round()
        m[N // 2] = N // 2
        h = torch.arange(N // 2 + 1, device="cuda", dtype=torch.float64)
        x = [h[None, None, :], m[None, :, None], m[:, None, None]]
        count = (x[0] != 0).int() + (x[1] != 0).int() + (x[2] != 0).int()
        self.xi = [torch.where((a == N // 2) & (count > 1), 0.0, a.expand(count.shape)) for a in x]
        n2 = self.xi[0] ** 2 + self.xi[1] ** 2 + self.xi[2] ** 2
        self.inv = torch.where(n2 > 0, 1.0 / n2.clamp(min=1.0), 0.0)

    def dot(self, s):
        return self.xi[0] * s[0] + self.xi[1] * s[1] + self.xi[2] * s[2]


def _sweeps(m, ph, e, n):
    N = ph.shape[0]
    k = torch.tensor(K3, dtype=torch.float64, device="cuda")[ph.long()]
    k0 = math.sqrt(min(K3) * max(K3))
    tau, eps = (k + k0) * e, []
    for _ in range(n):
        s = [torch.fft.rfftn((k - k0) / (k + k0) * t) for t in tau]
        d = m.dot(s) * m.inv
        new = torch.empty_like(tau)
        for c in range(3):
            s[c] -= 2 * m.xi[c] * d
            s[c][0, 0, 0] += 2 * k0 * E0[c] * N ** 3
            new[c] = torch.fft.irfftn(s[c], s=(N, N, N))
        eps.append(float((new - tau).norm()) / N ** 1.5 / (2 * k0) / np.linalg.norm(E0))
        tau = new
    return tau / (k + k0), eps


def _equilibrium(m, ph, e):
    N = ph.shape[0]
    phi = torch.tensor(K3, dtype=torch.float64, device="cuda")[ph.long()] * e
    flux = phi.mean(dim=(1, 2, 3)).cpu().numpy()
    a = m.dot([torch.fft.rfftn(p) for p in phi]).abs() ** 2
    tot = float(2 * a.sum() - a[..., 0].sum() - a[..., -1].sum())
    return 2 * math.pi / N * math.sqrt(tot) / N ** 3 / np.linalg.norm(flux), flux


@pytest.mark.parametrize("N", SIZES)
def test_sweeps_and_equilibrium(ctx, N):
    ph, e = _inputs(N)
    m = Modes(N)
    want, weps = _sweeps(m, ph, e, 2)
    weq, wflux = _equilibrium(m, ph, e)
    for prec, tol, rel in ((hmg.HMG_FP64, 2.0 ** -45, 2.0 ** -40), (hmg.HMG_FP32_BULK, 1e-5, 1e-4)):
        got = e.clone()
        torch.cuda.synchronize()
        eps = hmg.hmg_em_iterate(ctx.handle, ph, N, K3, E0, prec, 2, got)
        if prec == hmg.HMG_FP64:
            for c in range(3):
                assert float((got[c] - want[c]).norm()) < tol * float(want.norm())
        assert float((got - want).abs().max()) < max(tol, 1e-11) * float(want.abs().max())
        assert np.allclose(eps, weps, rtol=rel, atol=0)
        eq, flux = hmg.hmg_equilibrium(ctx.handle, ph, N, K3, prec, e)
        assert math.isclose(eq, weq, rel_tol=rel)
        assert np.abs(flux - wflux).max() < rel * np.abs(wflux).max()


@pytest.mark.parametrize("N", SIZES)
def test_forward_transform(ctx, N):
    _, e = _inputs(N)
    X = torch.empty_like(e)
    torch.cuda.synchronize()
    hmg.hmg_fft_forward(ctx.handle, N, 3, hmg.HMG_FP64, e, X)
    for c in range(3):
        h = torch.fft.rfftn(e[c])
        ref = h[..., :N // 2].clone()
        ref[..., 0] += 1j * h[..., N // 2]   # the kx = 0 entry packs the planes 0 and N/2
        got = torch.view_as_complex(X[c].reshape(N, N, N // 2, 2))
        assert float((got - ref).norm()) < 2.0 ** -47 * float(ref.norm())
