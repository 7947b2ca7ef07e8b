"""The work that users of libhmg have it do, as cases that can be timed and compared.

Each case is a dict of plain values; ``prepare`` makes what a program has in hand before the
call (device arrays, sphere lists and the one context it keeps), ``run`` makes one pass
through the public entry points of ``paper_1504_07499_gb300.hmg`` and ``exact`` gives the
same values from plain FP64 torch and numpy.  Sizes are the grids of §5 of the paper (64, 128,
256), of the benchmark configurations (32 to 512) and the other even 2^a 3^b sizes that the
entry points take.

FP32-bulk fields and FP32 sweeps are carried in double arrays by the C ABI; their values are
single-precision results, so ``run`` returns them as float32, as a program keeps them.
"""
import math

import numpy as np
import torch

from paper_1504_07499_gb300 import hmg, inputs

# every grid size the entry points take: even, 2^a 3^b, 8 .. 512
SIZES = sorted(n for a in range(1, 10) for b in range(0, 6) for n in [2 ** a * 3 ** b] if 8 <= n <= 512)
PREC = {"fp64": hmg.HMG_FP64, "fp32": hmg.HMG_FP32_BULK}
K_MATRIX, K_INCL = 0.20, 0.25     # with a coating of 2, 40 or 400: contrast 10, 200, 2000
TOL = 1e-8


def listed():
    return [
        # the smallest problem people start with: the plain FP64 method on a 32^3 grid with one
        # centred coated sphere, K and the gradient fields wanted (latency and launches count)
        dict(name="solve_fp64_sphere32", kind="solve", prec="fp64", N=32, n=1, f=4 * math.pi / 3 / 64, l=0.25, kc=400.0),
        # one realization at the paper's smallest routine resolution, contrast 2000
        dict(name="solve_bulk_64", kind="solve", prec="fp32", N=64, n=30, f=0.3, l=0.3, kc=400.0),
        # the benchmark problem: 256^3, 100 spheres, contrast 2000
        dict(name="solve_bulk_256", kind="solve", prec="fp32", N=256, n=100, f=0.3, l=0.3, kc=400.0),
        # the largest grid (the paper's cluster runs), at the contrast where it is routine
        dict(name="solve_bulk_512_c10", kind="solve", prec="fp32", N=512, n=100, f=0.3, l=0.3, kc=2.0),
        # the plain FP64 method as a check of a mid-size realization (a radix-3 grid, contrast 200)
        dict(name="solve_fp64_96_c200", kind="solve", prec="fp64", N=96, n=30, f=0.3, l=0.3, kc=40.0),
        # averaging over realizations of mixed sizes in one call (the request loop runs the same engine)
        dict(name="batch_mixed", kind="batch", n64=5, n96=4, n128=3, kc=400.0),
        # a program that drives the sweeps itself: FP32 arithmetic, one gradient
        dict(name="sweeps_fp32_192", kind="sweeps", prec="fp32", N=192, n=70, f=0.3, l=0.2, kc=400.0, n_iter=16),
        # the same in FP64 at the paper's finest routine resolution
        dict(name="sweeps_fp64_256", kind="sweeps", prec="fp64", N=256, n=100, f=0.3, l=0.2, kc=400.0, n_iter=4),
        # the equilibrium test of a field from elsewhere (another solver's result), on a 216^3 grid
        dict(name="equilibrium_fp64_216", kind="equilibrium", prec="fp64", N=216, n=70, f=0.3, l=0.3, kc=400.0),
        # the transforms by themselves, both directions, on a grid without kernels of its own
        dict(name="fft_fp32_144", kind="fft", prec="fp32", N=144, count=3),
        # sphere list -> phase grid at the finest routine resolution
        dict(name="voxelize_256", kind="voxelize", N=256, n=100, f=0.3, l=0.3),
        # a realization from its seed: placement (at 40 %, above the RSA jamming limit) and voxelization
        dict(name="rve_128", kind="rve", N=128, n=100, f=0.4, l=0.3),
    ]


def _sweeps(kc):
    """Sweeps per gradient that the contraction of the accelerated scheme asks for."""
    c = max(kc, K_INCL) / min(kc, K_MATRIX)
    rho = (math.sqrt(c) - 1) / (math.sqrt(c) + 1)
    return math.log(1 / TOL) / -math.log(rho)


def _log_size(rng, lo, hi):
    """A size of SIZES in [lo, hi], spread over the logarithm."""
    t = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((n for n in SIZES if lo <= n <= hi), key=lambda n: abs(math.log(n / t)))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batch", "sweeps", "sweeps", "equilibrium", "fft", "voxelize", "rve"])
    n = rng.randint(10, 100)
    geo = dict(n=n, f=round(rng.uniform(0.1, 0.3), 3), l=round(rng.uniform(0.1, 0.5), 3))
    kc = rng.choice([2.0, 40.0, 400.0])
    prec = rng.choice(["fp32", "fp32", "fp64"])
    if kind == "solve":
        # the plain FP64 method is drawn up to 96^3, the FP32-bulk one up to 256^3 at its own
        # sizes and up to 144^3 elsewhere, so that none costs more than the benchmark problem
        if prec == "fp64":
            N = _log_size(rng, 16, 96)
        else:
            N = _log_size(rng, 16, 256)
            if N > 144 and N not in (192, 256):
                N = 192 if N < 222 else 256
        return dict(kind=kind, prec=prec, N=N, kc=kc, **geo)
    if kind == "batch":
        return dict(kind=kind, n64=rng.randint(1, 6), n96=rng.randint(0, 4), n128=rng.randint(0, 3), kc=kc)
    if kind == "sweeps":
        return dict(kind=kind, prec=prec, N=_log_size(rng, 16, 256), kc=kc, n_iter=rng.randint(1, 16), **geo)
    if kind == "equilibrium":
        return dict(kind=kind, prec=prec, N=_log_size(rng, 16, 324), kc=kc, **geo)
    if kind == "fft":
        return dict(kind=kind, prec=prec, N=_log_size(rng, 8, 256), count=rng.randint(1, 6))
    if kind == "voxelize":
        return dict(kind=kind, N=_log_size(rng, 16, 512), **geo)
    return dict(kind=kind, N=_log_size(rng, 32, 256), n=n, f=round(rng.uniform(0.1, 0.4), 3), l=geo["l"])


# --- inputs ----------------------------------------------------------------------

_ctx = None


def _context():
    """The one context a program keeps for all its calls."""
    global _ctx
    if _ctx is None:
        _ctx = hmg.Context(0)
    return _ctx.handle


def _spheres(seed, n, f):
    """n identical spheres at volume fraction f by random sequential adsorption (one sphere: a
    radius of 1/4 and a centre near the middle of the cell)."""
    r = inputs.sphere_radius(n, f)
    if n == 1:
        c = 0.5 + 0.05 * (inputs.SplitMix64(seed).uniform(3).reshape(1, 3) - 0.5)
    else:
        c = None
        for s in range(20):   # RSA places these fractions; another stream if one should fail
            c = inputs.rsa(seed + 1_000_003 * s, n, r, max_candidates=400_000)
            if c is not None:
                break
    return np.ascontiguousarray(np.concatenate([c, np.full((n, 1), r)], axis=1))


def _phase(spheres, layer, N):
    """Three-phase grid of a sphere list (voxel centres, periodic), as torch gives it."""
    x = (torch.arange(N, device="cuda", dtype=torch.float32) + 0.5) / N
    outer = torch.zeros(N, N, N, dtype=torch.bool, device="cuda")
    core = torch.zeros_like(outer)
    for cx, cy, cz, r in spheres.tolist():
        d = []
        for c in (cx, cy, cz):
            a = (x - c % 1.0).abs()
            d.append(torch.minimum(a, 1 - a).square())
        yz = d[2][:, None] + d[1][None, :]
        rows = torch.nonzero(yz.reshape(-1) <= r * r).reshape(-1)   # (z, y) rows the sphere meets
        d2 = yz.reshape(-1)[rows][:, None] + d[0][None, :]
        outer.view(N * N, N)[rows] |= d2 <= r * r
        core.view(N * N, N)[rows] |= d2 <= ((1 - layer) * r) ** 2
    return torch.where(core, 1, torch.where(outer, 2, 0)).to(torch.uint8).contiguous()


def _gradient_field(seed, E, N):
    """E plus the gradient-like fluctuations of an unconverged solve: smooth and rough parts."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    e = torch.empty(3, N, N, N, dtype=torch.float64, device="cuda")
    x = torch.arange(N, device="cuda", dtype=torch.float64) * (2 * math.pi / N)
    for c in range(3):
        e[c].normal_(generator=g).mul_(0.3).add_(E[c])
        e[c] += 0.4 * torch.cos(x)[:, None, None] * torch.sin(2 * x)[None, :, None] * torch.cos(3 * x)[None, None, :]
    return e


def _batch_spec(case, seed):
    """(N, spheres, layer) of each RVE of a batch."""
    r = np.random.default_rng(seed)
    spec = []
    for N, cnt in ((64, case["n64"]), (96, case["n96"]), (128, case["n128"])):
        for _ in range(cnt):
            n, f = int(r.integers(10, 101)), float(r.uniform(0.1, 0.3))
            spec.append((N, _spheres(int(r.integers(1 << 40)), n, f), float(r.uniform(0.1, 0.5))))
    return spec


def _macro(seed):
    g = np.random.default_rng(seed).normal(size=3)
    return g / np.linalg.norm(g)


def prepare(case, seed):
    ctx = _context()
    s = dict(case, ctx=ctx)
    kind, N = case["kind"], case.get("N")
    if kind == "batch":
        spec = _batch_spec(case, seed)
        s["phases"] = [_phase(sp, l, n) for n, sp, l in spec]
        s["N_list"] = [n for n, _, _ in spec]
        s["k3"] = np.array([[K_MATRIX, K_INCL, case["kc"]]] * len(spec))
        return s
    if kind == "rve":
        s["seed"], s["r"] = seed, inputs.sphere_radius(case["n"], case["f"])
        s["phase"] = torch.empty(N, N, N, dtype=torch.uint8, device="cuda")
        s["spheres"] = np.empty((case["n"], 4))
        return s
    if kind == "fft":
        g = torch.Generator(device="cuda").manual_seed(seed)
        s["x"] = torch.randn(case["count"], N, N, N, dtype=torch.float64, device="cuda", generator=g)
        s["X"] = torch.empty(case["count"], N, N, N, dtype=torch.float64, device="cuda")   # N^2 N/2 complex
        s["y"] = torch.empty_like(s["x"])
        return s
    sph = _spheres(seed, case["n"], case["f"])
    if kind == "voxelize":
        s["spheres"] = sph
        s["phase"] = torch.empty(N, N, N, dtype=torch.uint8, device="cuda")
        return s
    s["phase"] = _phase(sph, case["l"], N)
    s["k"] = (K_MATRIX, K_INCL, case["kc"])
    if kind == "solve":
        s["e"] = torch.empty(3, 3, N, N, N, dtype=torch.float64, device="cuda")
    else:
        s["E"] = _macro(seed)
        s["e"] = _gradient_field(seed, s["E"], N)
    return s


# --- one pass ----------------------------------------------------------------------

def run(s):
    kind, N, ctx = s["kind"], s.get("N"), s["ctx"]
    if kind == "batch":
        K, _, _ = hmg.hmg_solve_batch(ctx, s["phases"], s["N_list"], s["k3"], TOL, hmg.HMG_FP32_BULK)
        return [K[i] for i in range(len(K))]
    if kind == "rve":
        gen = hmg.hmg_rve(ctx, s["seed"], s["n"], s["r"], s["l"], N, s["phase"], s["spheres"])
        return dict(generator=gen, phase=s["phase"], spheres=s["spheres"])
    if kind == "voxelize":
        hmg.hmg_voxelize(ctx, s["spheres"], s["l"], N, s["phase"])
        return s["phase"]
    prec = PREC[s["prec"]]
    out = (lambda t: t.float()) if s["prec"] == "fp32" else (lambda t: t)
    if kind == "fft":
        hmg.hmg_fft_forward(ctx, N, s["count"], prec, s["x"], s["X"])
        hmg.hmg_fft_inverse(ctx, N, s["count"], prec, s["X"], s["y"])
        return dict(X=out(s["X"]), y=out(s["y"]))
    if kind == "solve":
        K, _, _ = hmg.hmg_solve_fields(ctx, s["phase"], N, s["k"], TOL, prec, s["e"])
        return dict(K=K, e=out(s["e"]))
    if kind == "sweeps":
        eps = hmg.hmg_em_iterate(ctx, s["phase"], N, s["k"], s["E"], prec, s["n_iter"], s["e"])
        return dict(e=out(s["e"]), eps=eps.astype(np.float32) if s["prec"] == "fp32" else eps)
    eps, flux = hmg.hmg_equilibrium(ctx, s["phase"], N, s["k"], prec, s["e"])
    res = dict(eps=np.array([eps]), flux=flux)
    return {k: v.astype(np.float32) for k, v in res.items()} if s["prec"] == "fp32" else res


def work(case):
    kind, N = case["kind"], case.get("N")

    def fft(n):   # one real 3D transform
        return 2.5 * n ** 3 * 3 * math.log2(n)

    def sweeps(n, count, grads, word):
        # a sweep reads the field and the phases and writes the field; six 3D transforms and
        # about 40 pointwise operations per voxel
        return dict(bytes=count * grads * n ** 3 * (6 * word + 1.0), flops=count * grads * (6 * fft(n) + 40.0 * n ** 3))

    if kind == "batch":
        w = [sweeps(n, _sweeps(case["kc"]), 3, 4) for n in [64] * case["n64"] + [96] * case["n96"] + [128] * case["n128"]]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    if kind == "rve":
        return dict(bytes=N ** 3 + 64.0 * case["n"], flops=15.0 * N ** 3 + 10.0 * case["n"] ** 2 * 64)
    if kind == "voxelize":
        return dict(bytes=N ** 3 + 32.0 * case["n"], flops=15.0 * N ** 3)
    word = 4 if case["prec"] == "fp32" else 8
    if kind == "fft":
        return dict(bytes=case["count"] * N ** 3 * 32.0, flops=case["count"] * 2 * fft(N))
    if kind == "solve":
        return sweeps(N, _sweeps(case["kc"]), 3, word)
    if kind == "sweeps":
        return sweeps(N, case["n_iter"], 1, word)
    return dict(bytes=N ** 3 * 25.0, flops=3 * fft(N) + 20.0 * N ** 3)


# --- the same in 64 bits ------------------------------------------------------------

class _Grid:
    """Wavevectors and the projector of the half spectrum (kz, ky, kx <= N/2)."""

    def __init__(self, N):
        m = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64).round()
        m[N // 2] = N // 2
        h = torch.arange(N // 2 + 1, device="cuda", dtype=torch.float64)
        full = [h[None, None, :].expand(N, N, N // 2 + 1), m[None, :, None].expand(N, N, N // 2 + 1),
                m[:, None, None].expand(N, N, N // 2 + 1)]
        nonzero = sum((d != 0).to(torch.int32) for d in full)
        # Nyquist components count only where they are the only nonzero one
        self.xi = [torch.where((d == N // 2) & (nonzero > 1), 0.0, d) for d in full]
        n2 = sum(d * d for d in self.xi)
        self.inv = torch.where(n2 > 0, 1.0 / torch.where(n2 > 0, n2, 1.0), 0.0)
        self.weight = torch.full((N // 2 + 1,), 2.0, device="cuda", dtype=torch.float64)
        self.weight[0] = self.weight[N // 2] = 1.0
        self.N = N


def _em(grid, phase, k, E, e, n_iter, stop=0.0):
    """n_iter sweeps of the accelerated scheme on e (FP64); the residual of each sweep."""
    N = grid.N
    kk = torch.tensor(k, dtype=torch.float64, device="cuda")
    k0 = math.sqrt(min(k) * max(k))
    kv = kk[phase.long()]
    Y = (kv - k0) / (kv + k0)
    tau = (kv + k0) * e
    eps, nE = [], float(np.linalg.norm(E))
    for _ in range(n_iter):
        s = [torch.fft.rfftn(Y * tau[c]) for c in range(3)]
        dot = sum(grid.xi[c] * s[c] for c in range(3)) * grid.inv
        d2 = 0.0
        for c in range(3):
            t = s[c] - 2 * grid.xi[c] * dot
            t[0, 0, 0] += 2 * k0 * E[c] * N ** 3
            new = torch.fft.irfftn(t, s=(N, N, N))
            d2 = d2 + (new - tau[c]).square().sum()
            tau[c] = new
        eps.append(d2)
        if stop and len(eps) % 16 == 0 and math.sqrt(float(d2) / N ** 3) / (2 * k0) / nE < stop:
            break
    eps = [math.sqrt(float(d) / N ** 3) / (2 * k0) / nE for d in eps]
    return tau / (kv + k0), kv, eps


def _exact_solve(phase, k, fields):
    N = phase.shape[0]
    grid, K, es = _Grid(N), np.empty((3, 3)), []
    for j in range(3):
        E = np.eye(3)[j]
        e = torch.tensor(E, device="cuda").reshape(3, 1, 1, 1).expand(3, N, N, N).clone()
        e, kv, _ = _em(grid, phase, k, E, e, 1500, stop=1e-12)
        K[:, j] = (kv * e).mean(dim=(1, 2, 3)).cpu().numpy()
        if fields:
            es.append(e)
    return K, torch.stack(es) if fields else None


def _affordable(N, kc):
    """Whether torch solves this in about the time that is worth it."""
    return 3 * 1.6 * _sweeps(kc) * max(3e-4, N ** 3 * 1.5e-9) < 15.0


def exact(case, seed):
    kind, N = case["kind"], case.get("N")
    if kind in ("rve", "voxelize"):
        return None   # whole numbers and the placement's own stream
    if kind == "batch":
        out, spent = [], 0.0
        for n, sph, l in _batch_spec(case, seed):
            cost = 3 * 1.6 * _sweeps(case["kc"]) * max(3e-4, n ** 3 * 1.5e-9)
            if spent + cost < 12.0:
                spent += cost
                out.append(_exact_solve(_phase(sph, l, n), (K_MATRIX, K_INCL, case["kc"]), False)[0])
            else:
                out.append(None)
        return out
    if kind == "fft":
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn(case["count"], N, N, N, dtype=torch.float64, device="cuda", generator=g)
        X = torch.empty(case["count"], N, N, N // 2, dtype=torch.complex128, device="cuda")
        for i in range(case["count"]):
            h = torch.fft.rfftn(x[i])
            X[i] = h[..., :N // 2]
            X[i, ..., 0] += 1j * h[..., N // 2]   # the kx = 0 entry packs the planes 0 and N/2
        return dict(X=torch.view_as_real(X).reshape(case["count"], N, N, N), y=x * float(N) ** 3)
    phase = _phase(_spheres(seed, case["n"], case["f"]), case["l"], N)
    k = (K_MATRIX, K_INCL, case["kc"])
    if kind == "solve":
        if not _affordable(N, case["kc"]):
            return None
        K, e = _exact_solve(phase, k, True)
        return dict(K=K, e=e)
    E = _macro(seed)
    e = _gradient_field(seed, E, N)
    grid = _Grid(N)
    if kind == "sweeps":
        e, _, eps = _em(grid, phase, k, E, e, case["n_iter"])
        return dict(e=e, eps=np.array(eps))
    kv = torch.tensor(k, dtype=torch.float64, device="cuda")[phase.long()]
    flux = np.array([float((kv * e[c]).mean()) for c in range(3)])
    div = sum(grid.xi[c] * torch.fft.rfftn(kv * e[c]) for c in range(3))
    tot = float((grid.weight * (div.real.square() + div.imag.square())).sum())
    eps = 2 * math.pi / N * math.sqrt(tot) / N ** 3 / float(np.linalg.norm(flux))
    return dict(eps=np.array([eps]), flux=flux)
