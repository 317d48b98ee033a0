"""The workloads whose speed is measured, each through the package's public entry points.

Cubes are synthetic hyperspectral images made on the GPU: piecewise-constant abundances on Voronoi cells times
smooth spectra, scaled to [0, 1], with the mixed noise of the denoiser's setting (per-band Gaussian, impulses,
stripes, dead lines).  A cube of shape (n1, n2, n3) is a float32 tensor of shape (n3, n2, n1).
"""
import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_2204_12879_gb300 import lrstv
from paper_2204_12879_gb300.unrolled import UnrolledLRSTVFunction, default_theta

# shapes that uneven batches draw from (small test cubes, a mid size, the Indian Pines and Pavia shapes)
BATCH_SHAPES = ((64, 64, 31), (128, 128, 64), (145, 145, 220), (200, 200, 80))


def listed():
    return [
        # the operators a user composes into a penalty of their own, on a training-sized cube: launches and latency
        {"name": "gradient_64x64x31", "kind": "gradient", "n1": 64, "n2": 64, "n3": 31},
        # the same operators on a wide scene with a row length that is no multiple of four: memory traffic
        {"name": "gradient_511x512x191", "kind": "gradient", "n1": 511, "n2": 512, "n3": 191},
        # a Tikhonov-smoothed cube through the DFT-diagonalised solve, at the Indian Pines shape
        {"name": "zsolve_145x145x220", "kind": "zsolve", "n1": 145, "n2": 145, "n3": 220},
        # tensor-nuclear-norm shrinkage on its own (no earlier basis to start from): a patch ...
        {"name": "tsvt_64x64x31", "kind": "tsvt", "n1": 64, "n2": 64, "n3": 31, "level": 0.5},
        # ... and a long-spectrum patch with odd, unequal sides
        {"name": "tsvt_75x91x220", "kind": "tsvt", "n1": 75, "n2": 91, "n3": 220, "level": 0.4},
        # a whole denoise of a small cube: the smallest configuration, bound by launches
        {"name": "denoise_32x32x16", "kind": "denoise", "n1": 32, "n2": 32, "n3": 16, "iters": 20, "warm": True, "bf16x3": False},
        # a whole denoise of the Pavia-shaped cube: the benchmark's default workload
        {"name": "denoise_200x200x80", "kind": "denoise", "n1": 200, "n2": 200, "n3": 80, "iters": 50, "warm": True, "bf16x3": False},
        # the Washington-DC-shaped cube with the 3xBF16 products: the mixed-precision workload, stopped early as for a preview
        {"name": "denoise_256x256x191_bf16x3", "kind": "denoise", "n1": 256, "n2": 256, "n3": 191, "iters": 16, "warm": True, "bf16x3": True},
        # a scene with sides above 256 (tall Fourier slices), unequal
        {"name": "denoise_280x300x31", "kind": "denoise", "n1": 280, "n2": 300, "n3": 31, "iters": 12, "warm": True, "bf16x3": False},
        # uneven cubes denoised in lockstep, as a server batches its requests
        {"name": "batch_16_uneven", "kind": "batch", "cubes": 16, "pick": 5, "iters": 12},
        # one training step's forward and backward pass of the unrolled iteration, at its training size
        {"name": "unrolled_8x64x64x31", "kind": "unrolled", "n1": 64, "n2": 64, "n3": 31, "cubes": 8, "iters": 8},
        # the full model: Tucker projection inside the iteration, on a cube of low multilinear rank
        {"name": "tucker_64x60x31", "kind": "tucker", "n1": 64, "n2": 60, "n3": 31, "rank": 6, "iters": 10},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("gradient", "zsolve", "tsvt", "tsvt", "denoise", "denoise", "batch", "unrolled", "tucker"))
    if kind == "gradient":
        return {"kind": kind, "n1": log(32, 512), "n2": log(32, 512), "n3": log(8, 191)}
    if kind == "zsolve":
        return {"kind": kind, "n1": log(32, 256), "n2": log(32, 256), "n3": log(8, 220)}
    if kind == "tsvt":
        return {"kind": kind, "n1": log(24, 92), "n2": log(24, 92), "n3": log(8, 220), "level": round(rng.uniform(0.4, 0.6), 2)}
    if kind == "denoise":
        n1 = log(32, 280)
        n2 = min(300, max(32, int(round(n1 * rng.uniform(0.7, 1.4)))))
        tall, mixed = max(n1, n2) > 256, rng.random() < 0.3
        return {"kind": kind, "n1": n1, "n2": n2, "n3": log(8, 28 if tall else 96), "iters": rng.randint(8, 12 if tall or mixed else 50),
                "warm": tall or rng.random() < 0.8, "bf16x3": mixed}
    if kind == "batch":
        return {"kind": kind, "cubes": rng.randint(4, 12), "pick": rng.randint(6, 10 ** 6), "iters": rng.randint(8, 12)}
    if kind == "unrolled":
        n1 = rng.randint(24, 66)
        return {"kind": kind, "n1": n1, "n2": min(66, max(24, n1 + rng.randint(-12, 12))), "n3": rng.randint(12, 31),
                "cubes": rng.randint(2, 8), "iters": rng.randint(4, 8)}
    n1 = rng.randint(40, 66)
    return {"kind": kind, "n1": n1, "n2": min(66, max(40, n1 + rng.randint(-12, 12))), "n3": rng.randint(24, 40), "rank": rng.randint(3, 6),
            "iters": rng.randint(6, 10)}


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _cube(shape, g, sigma=(0.1, 0.2), impulse=0.2, stripes=0.3, dead=0.1, endmembers=6, cells=40, pair=False):
    """A noisy cube as an (n3, n2, n1) float32 tensor (pair: the clean cube beside it)."""
    n1, n2, n3 = shape

    def u(*s):
        return torch.rand(*s, generator=g, device="cuda")

    at, mix = u(cells, 2) * torch.tensor([n2, n1], device="cuda"), u(cells, endmembers) + 1e-3
    y, x = torch.meshgrid(torch.arange(n2, device="cuda"), torch.arange(n1, device="cuda"), indexing="ij")
    near = torch.full((n2, n1), math.inf, device="cuda")
    cell = torch.zeros((n2, n1), dtype=torch.long, device="cuda")
    for k in range(cells):
        d = (y - at[k, 0]) ** 2 + (x - at[k, 1]) ** 2
        cell = torch.where(d < near, k, cell)
        near = torch.minimum(d, near)
    abundance = (mix / mix.sum(1, keepdim=True))[cell]
    band = torch.arange(n3, device="cuda")[:, None, None]
    centre, width, height = u(endmembers, 3) * n3, (n3 / 20 + u(endmembers, 3) * n3 / 5).clamp(min=0.5), 0.2 + 0.8 * u(endmembers, 3)
    spectra = (height * torch.exp(-((band - centre) ** 2) / (2 * width ** 2))).sum(2)
    spectra = spectra / spectra.max(0, keepdim=True).values
    Y = clean = torch.einsum("jie,be->bji", abundance, spectra).contiguous()
    level = sigma[0] + (sigma[1] - sigma[0]) * u(n3, 1, 1)
    Y = Y + level * torch.randn(n3, n2, n1, generator=g, device="cuda")
    hit = u(n3, n2, n1) < impulse
    Y = torch.where(hit, (u(n3, n2, n1) < 0.5).float(), Y)
    striped = (u(n3, 1, 1) < stripes) & (u(n3, n2, 1) < 0.1)
    Y = Y + striped * (0.5 * u(n3, n2, 1) - 0.25)
    gone = (u(n3, 1, 1) < dead) & (u(n3, n2, 1) < 0.05)
    Y = torch.where(gone, torch.zeros_like(Y), Y).contiguous()
    return (Y, clean) if pair else Y


def _batch(case):
    """The shapes and noise levels of a batch: uneven cubes, each with noise of its own."""
    r = np.random.RandomState(case["pick"])
    return [(BATCH_SHAPES[int(r.randint(len(BATCH_SHAPES)))], float(r.uniform(0.05, 0.2)), float(r.uniform(0.0, 0.3)))
            for _ in range(case["cubes"])]


def _shape(case):
    return case["n1"], case["n2"], case["n3"]


def _flags(case):
    return (lrstv.FLAG_WARM_START if case["warm"] else 0) | (lrstv.FLAG_BF16X3 if case["bf16x3"] else 0)


def _params(case):
    return lrstv.Params.make(case["n1"], case["n2"], max_iter=case["iters"], flags=_flags(case))


def _low_rank(shape, r, g):
    """A cube of multilinear rank (r, r, r), its leading values well apart from the noise."""
    n1, n2, n3 = shape
    U = [torch.linalg.qr(torch.randn(n, r, generator=g, device="cuda", dtype=torch.float64))[0] for n in (n3, n2, n1)]
    s = math.sqrt(n1 * n2 * n3) * torch.cat([torch.tensor([0.5], dtype=torch.float64), torch.linspace(0.2, 0.1, r - 1, dtype=torch.float64)])
    Y = torch.einsum("k,ak,bk,ck->abc", s.cuda(), *U) + 0.02 * torch.randn(n3, n2, n1, generator=g, device="cuda", dtype=torch.float64)
    return Y.float().contiguous()


def _tsvt_input(case, g):
    """A gradient map of a noisy cube and a threshold of `level` times the edge of its noise's singular values."""
    Y = _cube(_shape(case), g)
    A = (torch.roll(Y, -1, 2) - Y).contiguous()
    return A, float(np.float32(case["level"] * math.sqrt(case["n3"] * max(case["n1"], case["n2"])) * float(A.std())))


def prepare(case, seed):
    g, kind = _generator(seed), case["kind"]
    state = {"kind": kind, "case": case}
    if kind == "batch":
        cubes = _batch(case)
        shapes = [c[0] for c in cubes]
        params = [lrstv.Params.make(s[0], s[1], max_iter=case["iters"], flags=lrstv.FLAG_WARM_START) for s in shapes]
        state["Y"] = [_cube(s, g, (sig, sig), imp, 0.0, 0.0, 6, 24) for s, sig, imp in cubes]
        state["batch"] = lrstv.Batch(shapes, params)
        return state
    shape = _shape(case)
    if kind in ("gradient", "zsolve"):
        state["Y"] = _cube(shape, g)
    elif kind == "tsvt":
        state["Y"], state["t"] = _tsvt_input(case, g)
    elif kind == "denoise":
        state["Y"] = _cube(shape, g)
        state["plan"] = lrstv.Plan(*shape, _params(case))
    elif kind == "tucker":
        state["Y"] = _low_rank(shape, case["rank"], g)
        state["plan"] = lrstv.Plan(*shape, lrstv.Params.make(shape[0], shape[1], max_iter=case["iters"], flags=lrstv.FLAG_WARM_START))
        state["plan"].set_tucker((case["rank"],) * 3)
    else:
        pairs = [_cube(shape, g, (0.1, 0.1), 0.1, 0.0, 0.0, 4, 12, pair=True) for _ in range(case["cubes"])]
        state["Y"], state["clean"] = (torch.stack(x) for x in zip(*pairs))
        state["theta"] = torch.tensor(default_theta(shape[0], shape[1], case["iters"]), dtype=torch.float32,
                                      device="cuda", requires_grad=True)
        state["handle"] = lrstv.Unroll(shape, case["cubes"], case["iters"], flags=lrstv.FLAG_WARM_START)
    return state


def run(state):
    kind, case, Y = state["kind"], state["case"], state["Y"]
    if kind == "batch":
        X, S = state["batch"].run(Y)
        return {"X": X, "S": S}
    shape = _shape(case)
    if kind == "gradient":
        gmap = lrstv.lrstv_diff(Y, shape, (1.0, 1.0, 0.5))
        cut = lrstv.lrstv_soft_threshold(gmap, 0.1)
        return {"gradient": gmap, "cut": cut, "adjoint": lrstv.lrstv_diff_adjoint(cut, shape, (1.0, 1.0, 0.5))}
    if kind == "zsolve":
        return lrstv.lrstv_zsolve(Y, shape, 0.7)
    if kind == "tsvt":
        return lrstv.lrstv_tsvt(Y, shape, state["t"])
    if kind == "unrolled":
        theta = state["theta"]
        theta.grad = None
        X = UnrolledLRSTVFunction.apply(Y, theta, state["handle"])
        torch.nn.functional.mse_loss(X, state["clean"]).backward()
        return {"X": X.detach(), "dtheta": theta.grad}
    X, S = state["plan"].run(Y)
    return {"X": X, "S": S}


def _iteration_work(n1, n2, n3):
    """Bytes and operations of one iteration: 18 state cubes read and 15 written; the DFTs of one Z-solve and of
    three t-SVTs as products with the DFT matrices; one sweep of column inner products and the two products that
    apply an SVD's factors, on half the Fourier slices (the others are their conjugates)."""
    N, h, nr, nc = n1 * n2 * n3, n3 // 2 + 1, max(n1, n2), min(n1, n2)
    dft = 4.0 * 2 * n3 * h * n1 * n2 * 4
    spatial = 8.0 * 2 * h * n1 * n2 * (n1 + n2)
    svd = 3.0 * h * (8.0 * nr * nc * nc / 2 + 2 * 8.0 * nr * nc * nc)
    return 4.0 * 33 * N, dft + spatial + svd


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0.0
        for s, _, _ in _batch(case):
            x, y = _iteration_work(*s)
            b, f = b + x * case["iters"], f + y * case["iters"]
        return {"bytes": b, "flops": f}
    n1, n2, n3 = _shape(case)
    N, h, nr, nc = n1 * n2 * n3, n3 // 2 + 1, max(n1, n2), min(n1, n2)
    if kind == "gradient":
        return {"bytes": 4.0 * 14 * N, "flops": 18.0 * N}
    if kind == "zsolve":
        return {"bytes": 8.0 * N, "flops": 2.0 * 4 * n3 * h * n1 * n2 / 2 + 8.0 * 2 * h * n1 * n2 * (n1 + n2)}
    if kind == "tsvt":  # an SVD of each slice of half the spectrum (about 30 nr nc^2 real operations) and the product of its factors
        return {"bytes": 8.0 * N, "flops": 2.0 * 4 * n3 * h * n1 * n2 / 2 + h * (30.0 + 8.0) * nr * nc * nc}
    b, f = _iteration_work(n1, n2, n3)
    k = case["iters"] * (3 * case["cubes"] if kind == "unrolled" else 1)  # a backward pass takes about twice its forward pass
    return {"bytes": b * k, "flops": f * k}


# ---------------------------------------------------------------- in 64 bits
def _svt(slices, t):
    """Singular values of each matrix of a list shrunk by t."""
    def one(M):
        U, s, Vh = np.linalg.svd(M, full_matrices=False)
        return (U * np.maximum(s - t, 0.0)) @ Vh

    with ThreadPoolExecutor(8) as ex:
        return list(ex.map(one, slices))


def _tsvt(A, t):
    """A: (m, n3, n2, n1) float64; the t-SVT of each of the m cubes."""
    A = np.asarray(A)
    m, n3 = A.shape[:2]
    spec = np.fft.rfft(A, axis=1)
    out = _svt([spec[i, k] for i in range(m) for k in range(spec.shape[1])], t)
    return np.fft.irfft(np.stack(out).reshape(spec.shape), n=n3, axis=1)


def _soft(x, d):
    return np.sign(x) * np.maximum(np.abs(x) - d, 0.0)


_AXES = (2, 1, 0)  # mode n of a cube is axis _AXES[n] of its (n3, n2, n1) array


def _diff(x):
    return np.stack([np.roll(x, -1, a) - x for a in _AXES])


def _adjoint(g):
    return sum(np.roll(g[n], 1, a) - g[n] for n, a in enumerate(_AXES))


def _solve(T, mu):
    P = 0.0
    for a in range(3):
        n = T.shape[a]
        P = P + (4.0 * np.sin(np.pi * np.arange(n) / n) ** 2).reshape([-1 if b == a else 1 for b in range(3)])
    return np.fft.ifftn(np.fft.fftn(T) / (mu * (1.0 + P))).real


def _admm(Y, scalars):
    """Algorithm 1 from L = Z = Y with (tau, alpha, lambda, mu) of each iteration; returns L and S."""
    L, Z, S = Y.copy(), Y.copy(), np.zeros_like(Y)
    G1, G2 = np.zeros_like(Y), np.zeros_like(Y)
    F, E, G3, G4 = (np.zeros((3,) + Y.shape) for _ in range(4))
    for tau, alpha, lam, mu in scalars:
        L = 0.5 * (Y - S + Z + (G1 - G2) / mu)
        Z = _solve(mu * L + G2 + _adjoint(mu * F - G3), mu)
        D = _diff(Z)
        F = _soft(0.5 * (D + G3 / mu + E + G4 / mu), tau / mu)
        S = _soft(Y - L + G1 / mu, lam / mu)
        G1 = G1 + mu * (Y - L - S)
        G2 = G2 + mu * (L - Z)
        G3 = G3 + mu * (D - F)
        E = _tsvt(F - G4 / mu, alpha / mu)
        G4 = G4 + mu * (E - F)
    return L, S


def _host(t):
    return t.detach().double().cpu().numpy()


def exact(case, seed):
    kind, g = case["kind"], _generator(seed)
    if kind in ("batch", "tucker"):
        return None
    n1, n2, n3 = shape = _shape(case)
    nr, nc, h = max(n1, n2), min(n1, n2), n3 // 2 + 1
    if kind == "gradient":
        Y, w = _cube(shape, g), (1.0, 1.0, 0.5)
        Y = Y.double()
        gmap = torch.stack([c * (torch.roll(Y, -1, a) - Y) for c, a in zip(w, _AXES)])
        cut = torch.sign(gmap) * torch.clamp(gmap.abs() - float(np.float32(0.1)), min=0.0)
        back = sum(c * (torch.roll(cut[n], 1, a) - cut[n]) for n, (c, a) in enumerate(zip(w, _AXES)))
        return {"gradient": gmap.reshape(-1), "cut": cut.reshape(-1), "adjoint": back.reshape(-1)}
    if kind == "zsolve":
        return _solve(_host(_cube(shape, g)), float(np.float32(0.7))).reshape(-1)
    if kind == "tsvt":
        A, t = _tsvt_input(case, g)
        return _tsvt(_host(A)[None], t)[0].reshape(-1)
    svds = 3.0 * h * case["iters"] * nr * nc * nc
    if kind == "denoise":
        if svds > 6e8 or case["bf16x3"]:
            return None
        p = _params(case)
        mu, scalars = float(p.mu0), []
        for _ in range(case["iters"]):
            scalars.append((float(p.tau), float(p.alpha), float(p.lam), mu))
            mu = min(float(p.rho) * mu, float(p.mu_max))
        X, S = _admm(_host(_cube(shape, g)), scalars)
        return {"X": X.reshape(-1), "S": S.reshape(-1)}
    if svds * case["cubes"] > 2e9:
        return None
    scalars = torch.tensor(default_theta(n1, n2, case["iters"]), dtype=torch.float32).double().tolist()
    X = [_admm(_host(_cube(shape, g, (0.1, 0.1), 0.1, 0.0, 0.0, 4, 12)), scalars)[0] for _ in range(case["cubes"])]
    return {"X": np.stack(X), "dtheta": None}
