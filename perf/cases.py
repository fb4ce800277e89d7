"""Timed cases of the library's public entry points.

A case is one call, or one chain of calls, of paper_2510_26574_gb300 as a user's
program makes them: the partial Cholesky factor (greedy or randomly pivoted, FP64 or
the precision form), the normalisation, the top-k eigenpairs, the batched factors,
the low-memory form and the symmetric normalisation.  `prepare` makes the points (and
the factor, where a call takes one) on the GPU from a seed, `run` is one pass, `work`
states the bytes and operations no implementation can do without, and `exact` gives the
same outputs from plain torch in 64 bits.

Points: Kuramoto-Sivashinsky states (u_t = -u u_x - u_xx - u_xxxx, L = 22, 64 modes,
ETDRK4 with dt = 0.25, samples 1.0 apart), their delay embeddings at one grid point,
or Gaussian mixtures around such states.  The bandwidth is the median squared distance.
"""
import math

import numpy as np
import torch

import paper_2510_26574_gb300 as kevd

DEV = "cuda:0"
F64, F32 = torch.float64, torch.float32


def listed():
    return [
        # the smallest problem a user decomposes: one trajectory, greedy pivots, all three
        # stages; launches and latency count
        dict(name="greedy_whole_2k", form="whole", mode="greedy", prec="fp64", points="ks", N=2000, d=64, r=128, b=1,
             k=32),
        # the plain FP64 factor at its usual size
        dict(name="factor_fp64_200k", form="factor", mode="arpc", prec="fp64", points="ks", N=200000, d=64, r=1024,
             b=64, k=0),
        # the FP64 factor of a large space-time embedding (the precision form's counterpart)
        dict(name="factor_fp64_1m", form="factor", mode="arpc", prec="fp64", points="vsa", N=1000000, d=128, r=2048,
             b=128, k=0),
        # degree vectors and Grams of a stored FP64 factor, rank as an ARPC run leaves it
        dict(name="normalize_fp64_256k", form="normalize", mode="", prec="fp64", points="vsa", N=262144, d=128, r=1101,
             b=0, k=0),
        # the same call on one problem of a batch of uneven sizes: odd N, small rank
        dict(name="normalize_fp64_odd", form="normalize", mode="", prec="fp64", points="ks", N=60001, d=64, r=401, b=0,
             k=0),
        # top-64 eigenpairs from an FP64 factor and its Grams
        dict(name="eig_fp64_200k", form="eig", mode="", prec="fp64", points="ks", N=200000, d=64, r=801, b=0, k=64),
        # the precision form's factor on the two space-time embeddings
        dict(name="factor_bf16x3_524k", form="factor", mode="arpc", prec="bf16x3", points="vsa", N=524288, d=96, r=2048,
             b=128, k=0),
        dict(name="factor_bf16x3_2m", form="factor", mode="arpc", prec="bf16x3", points="vsa", N=2000000, d=128, r=2048,
             b=128, k=0),
        # degree vectors and Grams of the large FP32 factor
        dict(name="normalize_bf16x3_2m", form="normalize", mode="", prec="bf16x3", points="vsa", N=2000000, d=128,
             r=1848, b=0, k=0),
        # top-128 eigenpairs from an FP32 factor and its Grams
        dict(name="eig_bf16x3_524k", form="eig", mode="", prec="bf16x3", points="vsa", N=524288, d=96, r=1661, b=0,
             k=128),
        # many small independent problems of uneven N, d, eps and r in one launch
        dict(name="batch_16", form="batch", mode="arpc", prec="fp64", points="mix", N=100000, d=0, r=512, b=64, k=16),
        # the factor too large to store: pivots and an r x r block only, then the Grams
        dict(name="lowmem_60k", form="lowmem", mode="arpc", prec="fp64", points="ks", N=60000, d=64, r=512, b=64, k=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    form = rng.choice(["factor", "factor", "factor", "normalize", "normalize", "eig", "whole", "batch", "lowmem",
                       "symmetric"])
    prec = rng.choice(["fp64", "bf16x3"])
    points = rng.choice(["ks", "vsa", "vsa"])
    d = 64 if points == "ks" else rng.choice([32, 64, 77, 96, 128])
    c = dict(form=form, mode="", prec=prec, points=points, N=0, d=d, r=0, b=0, k=0)
    if form == "factor":
        c["mode"] = "arpc"
        c["N"] = _log(rng, 2000, 1000000 if prec == "fp64" else 2000000)
        c["r"] = _log(rng, 64, min(2048, c["N"] // 8))
        c["b"] = min(rng.choice([16, 32, 48, 64, 100, 128]), c["r"])
        if c["b"] < 32:     # the FP64-pipe engine's flops
            c["N"] = min(c["N"], 100000)
            c["r"] = min(c["r"], 512, c["N"] // 8)
            c["b"] = min(c["b"], c["r"])
    elif form in ("normalize", "eig", "symmetric"):
        c["N"] = _log(rng, 2000, 260000 if prec == "fp64" else 1000000)
        c["r"] = _log(rng, 64, min(1100 if prec == "fp64" else 1800, c["N"] // 8))
        if c["N"] % 2 and prec == "fp64":
            c["r"] = min(c["r"], int(math.sqrt(5e10 / c["N"])))
        c["k"] = {"normalize": 0, "eig": min(rng.choice([16, 32, 64]), c["r"] // 4), "symmetric": 16}[form]
    elif form == "whole":
        c.update(mode="greedy", prec="fp64", N=_log(rng, 500, 20000), b=1)
        c["r"] = _log(rng, 32, min(256, c["N"] // 8))
        c["k"] = min(rng.choice([8, 16, 32]), c["r"] // 4)
    elif form == "batch":
        c.update(mode="arpc", prec="fp64", points="mix", N=_log(rng, 8000, 100000), d=0, r=_log(rng, 160, 512),
                 b=rng.choice([32, 64]), k=rng.randint(4, 16))
    else:
        c.update(mode="arpc", prec="fp64", N=_log(rng, 4000, 60000))
        c["r"] = _log(rng, 64, min(512, c["N"] // 8))
        c["b"] = min(rng.choice([32, 64]), c["r"])
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _ks(traj, samples, seed):
    """(traj, samples, 64) grid values: ETDRK4 steps of `traj` trajectories at once, each from
    its own seeded state of amplitude 0.1, spun up for 100 time units."""
    L, M, h = 22.0, 64, 0.25
    q = 2 * np.pi / L * np.arange(M // 2)
    lin = q ** 2 - q ** 4
    z = h * lin[:, None] + np.exp(1j * np.pi * (np.arange(1, 33) - 0.5) / 32)[None, :]

    def mean(v):
        return torch.from_numpy(h * np.real(np.mean(v, axis=1))).to(DEV)

    E, E2 = (torch.from_numpy(np.exp(a * h * lin)).to(DEV) for a in (1.0, 0.5))
    Q = mean((np.exp(z / 2) - 1) / z)
    f1 = mean((-4 - z + np.exp(z) * (4 - 3 * z + z ** 2)) / z ** 3)
    f2 = 2 * mean((2 + z + np.exp(z) * (-2 + z)) / z ** 3)
    f3 = mean((-4 - 3 * z - z ** 2 + np.exp(z) * (4 - z)) / z ** 3)
    g = torch.from_numpy(-0.5j * q).to(DEV)

    def nonlin(v):
        u = torch.fft.irfft(v, n=96, norm="forward")        # zero padded: 3/2 dealiasing
        return g * torch.fft.rfft(u * u, norm="forward")[..., : M // 2]

    gen = torch.Generator().manual_seed(seed)
    u0 = 0.1 * torch.randn(traj, M, generator=gen, dtype=F64).to(DEV)
    v = torch.fft.rfft(u0 - u0.mean(1, keepdim=True), norm="forward")[:, : M // 2].contiguous()
    out = torch.empty(traj, samples, M, dtype=F64, device=DEV)
    for j in range(samples):
        for _ in range(400 if j == 0 else 4):
            nv = nonlin(v)
            ev = E2 * v
            a = ev + Q * nv
            na = nonlin(a)
            nb = nonlin(ev + Q * na)
            nc = nonlin(E2 * a + Q * (2 * nb - nv))
            v = E * v + nv * f1 + (na + nb) * f2 + nc * f3
        out[:, j] = torch.fft.irfft(v, n=M, norm="forward")
    return out


def _median(X, seed):
    gen = torch.Generator().manual_seed(seed + 1)
    i, j = (torch.randint(X.shape[0], (1 << 15,), generator=gen).to(DEV) for _ in range(2))
    d2 = (X[i].double() - X[j].double()).square().sum(1)
    return float(d2[d2 > 0].median())


def _points(case, seed, dtype):
    N, d = case["N"], case["d"]
    if case["points"] == "ks":
        per = 100
        X = _ks(-(-N // per), per, seed).reshape(-1, 64)[:N]
    else:                                                    # d delays at one grid point
        per = 125
        u = _ks(-(-N // (64 * per)), per + d - 1, seed).to(dtype)
        X = u.unfold(1, d, 1).flip(-1).reshape(-1, d)[:N]
    X = X.to(dtype).contiguous()
    return X, _median(X, seed)


def _factor(X, eps, r, seed):
    """A rank-r factor of the kernel matrix as the eigen stage receives it: K(:, S) L^-T for r
    random distinct pivots, an (r, N) tensor of X's type."""
    gen = torch.Generator().manual_seed(seed + 2)
    S = torch.randperm(X.shape[0], generator=gen)[:r].to(DEV)
    XS = X[S].double()
    L = torch.linalg.cholesky(_kernel(XS, XS, eps) + 1e-7 * torch.eye(r, dtype=F64, device=DEV))
    Linv = torch.linalg.solve_triangular(L, torch.eye(r, dtype=F64, device=DEV), upper=False).to(X.dtype)
    F = torch.empty(r, X.shape[0], dtype=X.dtype, device=DEV)
    XS = XS.to(X.dtype)
    for c in range(0, X.shape[0], 1 << 18):
        F[:, c:c + (1 << 18)] = Linv @ _kernel(XS, X[c:c + (1 << 18)], eps)
    return F


def _kernel(A, B, eps):
    d2 = (A * A).sum(1)[:, None] + (B * B).sum(1)[None, :] - 2.0 * (A @ B.T)
    return torch.exp_(d2.clamp_(min=0.0).mul_(-1.0 / eps))


def _grams(F, weights):
    """F diag(w) F^T for each w, an (r, N) factor in blocks of rows: products in F's type,
    sums over blocks in 64 bits; upper blocks, mirrored."""
    r, N = F.shape
    out = [torch.zeros(r, r, dtype=F64, device=DEV) for _ in weights]
    step = 1 << 14 if F.dtype == F32 else 1 << 16
    for c in range(0, N, step):
        f = F[:, c:c + step]
        for G, w in zip(out, weights):
            fw = f * w[c:c + step].to(F.dtype)
            for j in range(0, r, 512):
                G[j:j + 512, j:] += fw[j:j + 512] @ f[j:].T
    return [torch.triu(G) + torch.triu(G, 1).T for G in out]


def _degrees(F):
    s = torch.zeros(F.shape[0], dtype=F64, device=DEV)
    N, step = F.shape[1], 1 << 18
    cut = [slice(c, c + step) for c in range(0, N, step)]
    for c in cut:
        s += F[:, c].double().sum(1)
    d = torch.cat([s @ F[:, c].double() for c in cut])
    t = torch.zeros_like(s)
    for c in cut:
        t += F[:, c].double() @ (1.0 / d[c])
    q = torch.cat([t @ F[:, c].double() for c in cut])
    return d, q


def _problems(case, seed):
    """k problems with N up to case N and r up to case r: mixtures of eight Gaussians around
    KS states, d in {32, 64, 128}, eps a multiple of the median squared distance."""
    rng = np.random.Generator(np.random.PCG64([case["N"], case["r"], case["k"]]))
    u = _ks(case["k"], 9, seed)
    probs = []
    for p in range(case["k"]):
        N = int(rng.integers(case["N"] // 20, case["N"] + 1))
        d = int(rng.choice([32, 64, 128]))
        r = int(rng.integers(case["r"] // 4, case["r"] + 1))
        r = max(case["b"], min(r, N // 2))
        s = u[p]
        means = s[:8, ::2] if d == 32 else s[:8] if d == 64 else torch.cat([s[:8], s[1:9]], 1)
        sep = torch.cdist(means, means).square().sum().div(56).sqrt()
        gen = torch.Generator().manual_seed(seed * 1000 + p)
        comp = torch.randint(8, (N,), generator=gen).to(DEV)
        X = means[comp] + 0.1 * sep * torch.randn(N, d, generator=gen, dtype=F64).to(DEV)
        eps = float(rng.choice([0.25, 0.5, 1.0, 2.0])) * _median(X, p)
        probs.append(dict(X=X.contiguous(), eps=eps, r=r, b=case["b"], seed=2000 + p))
    return probs


def prepare(case, seed):
    s = dict(case=case, seed=seed % (1 << 31))
    form, dtype = case["form"], F64 if case["prec"] == "fp64" else F32
    if form == "batch":
        s["batch"] = kevd.Batch(_problems(case, s["seed"]))
        return s
    s["X"], s["eps"] = _points(case, s["seed"], dtype)
    if form in ("normalize", "eig", "symmetric"):
        s["F"] = _factor(s.pop("X"), s["eps"], case["r"], s["seed"])
    if form == "eig":
        s["d"], q = _degrees(s["F"])
        s["A"], s["C"] = _grams(s["F"], [1.0 / (s["d"] * s["d"]), 1.0 / q])
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _pivots(o):
    """The pivots of a call that allocates r entries and fills `rank`: the rest is marked."""
    o["pivots"][o["rank"]:] = -1
    return o["pivots"]


def run(s):
    c = s["case"]
    form = c["form"]
    tau = 1e-13 if c["prec"] == "fp64" else 1e-6
    if form == "normalize":
        return kevd.bistoch_normalize(s["F"], c["r"])
    if form == "eig":
        return kevd.eig_topk(s["F"], c["r"], s["d"], s["A"], s["C"], c["k"], tau=tau)
    if form == "symmetric":
        d, As = kevd.symmetric_normalize(s["F"], c["r"])
        return d, As, kevd.symmetric_eig_topk(s["F"], c["r"], d, As, c["k"])
    if form == "batch":
        out = s["batch"].run()
        return [dict(F=o["F"], rho=o["rho"], pivots=_pivots(o)) for o in out]
    if form == "lowmem":
        o = kevd.rpchol_factor_lowmem(s["X"], s["eps"], c["r"], b=c["b"], seed=s["seed"])
        d, q, A, C = kevd.bistoch_normalize_lowmem(s["X"], s["eps"], o["pivots"], o["W"], o["rank"])
        pad = (0, c["r"] - o["rank"]) * 2
        return dict(W=o["W"], rho=o["rho"], pivots=_pivots(o), trace_err=o["trace_err"], d=d, q=q,
                    A=torch.nn.functional.pad(A, pad), C=torch.nn.functional.pad(C, pad))
    o = kevd.rpchol_factor(s["X"], s["eps"], c["r"], mode=c["mode"], b=c["b"], seed=s["seed"])
    out = dict(F=o["F"], rho=o["rho"], pivots=_pivots(o), trace_err=o["trace_err"])
    if form == "whole":
        d, q, A, C = kevd.bistoch_normalize(o["F"], o["rank"])
        ev, U, _ = kevd.eig_topk(o["F"], o["rank"], d, A, C, c["k"])
        out.update(d=d, q=q, A=A, C=C, ev=ev, U=U)
    return out


def work(case):
    N, d, r, k = case["N"], case["d"], case["r"], case["k"]
    e = 8 if case["prec"] == "fp64" else 4
    form = case["form"]
    if form == "batch":     # N and r are upper ends of uniform ranges
        n, rr, dd = 0.525 * N * k, 0.625 * r, 75
        return dict(bytes=8 * n * (dd + rr + 1), flops=n * (2 * dd * rr + rr * rr))
    if form == "lowmem":
        return dict(bytes=8 * (N * (d + 3) + 3 * r * r), flops=N * (2 * d * r + r * r + 2 * r * (r + 1)))
    factor = dict(bytes=e * N * (d + r) + 8 * N, flops=N * (2 * d * r + r * r))
    norm = dict(bytes=e * N * r + 16 * N + 16 * r * r, flops=N * (8 * r + 2 * r * (r + 1)))
    eig = dict(bytes=e * N * r + 8 * N * (k + 1) + 16 * r * r, flops=2 * N * r * k + 6 * r ** 3)
    if form == "symmetric":
        return dict(bytes=2 * e * N * r + 8 * N * (k + 2), flops=N * (4 * r + r * (r + 1) + 2 * r * k) + 4 * r ** 3)
    parts = {"factor": [factor], "normalize": [norm], "eig": [eig], "whole": [factor, norm, eig]}[form]
    return {w: sum(p[w] for p in parts) for w in ("bytes", "flops")}


# ---------------------------------------------------------------------------
# the same outputs in 64 bits, plain torch and numpy
# ---------------------------------------------------------------------------
def _philox(seed, stream, rnd, n):
    """Uniforms of Philox4x32-10 with key = seed and counters (j, rnd, stream, 0)."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [np.arange(n, dtype=np.uint64), np.full(n, rnd, np.uint64), np.full(n, stream, np.uint64),
         np.zeros(n, np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for i in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1),
             p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return ((c[0] >> np.uint64(5)).astype(np.float64) * 67108864.0 + (c[1] >> np.uint64(6)).astype(np.float64)) / 2.0 ** 53


def _reject(H, z):
    H = H.copy()
    T, L, rho0 = [], np.zeros_like(H), np.diag(H).copy()
    for i in range(H.shape[0]):
        if H[i, i] > 0 and z[i] * rho0[i] < H[i, i]:
            T.append(i)
            L[i:, i] = H[i:, i] / math.sqrt(H[i, i])
            H[i + 1:, i + 1:] -= np.outer(L[i + 1:, i], L[i + 1:, i])
    return T, L[np.ix_(T, T)]


def _pchol(X, eps, r, mode, b, seed):
    """Algorithm 2 (or greedy pivots): F as an (r, N) tensor, rho, pivots."""
    N = X.shape[0]
    F = torch.zeros(r, N, dtype=F64, device=DEV)
    rho = torch.ones(N, dtype=F64, device=DEV)
    piv = []
    for rnd in range(r if mode == "greedy" else r // b):
        if mode == "greedy":
            prop = torch.nonzero(rho == rho.max())[:1, 0]
        else:
            cs = torch.cumsum(rho, 0)
            u = torch.from_numpy(_philox(seed, 0, rnd, b)).to(DEV)
            prop = torch.searchsorted(cs, u * cs[-1], right=True).clamp(max=N - 1)
        k = len(piv)
        FS = F[:k, prop]
        Kp = _kernel(X[prop], X[prop], eps)
        Kp[prop[:, None] == prop[None, :]] = 1.0
        H = (Kp - FS.T @ FS).cpu().numpy()
        if mode == "greedy":
            T, L = ([0], np.sqrt(H)) if H[0, 0] > 0 else ([], None)
        else:
            T, L = _reject(H, _philox(seed, 1, rnd, b))
        if not T:
            if mode == "greedy":
                break
            continue
        acc = prop[torch.tensor(T, device=DEV)]
        Kc = _kernel(X[acc], X, eps)
        Kc[torch.arange(len(T), device=DEV), acc] = 1.0
        R = Kc - F[:k, acc].T @ F[:k]
        G = torch.linalg.solve_triangular(torch.from_numpy(L).to(DEV), R, upper=False)
        F[k:k + len(T)] = G
        rho = (rho - G.square().sum(0)).clamp(min=0.0)
        piv += acc.tolist()
    return F, rho, torch.tensor(piv, dtype=torch.int64)


def _norm_exact(F):
    d, q = _degrees(F)
    A, C = _grams64(F, [1.0 / (d * d), 1.0 / q])
    return d, q, A, C


def _grams64(F, weights):
    """_grams with 64-bit products."""
    out = [torch.zeros(F.shape[0], F.shape[0], dtype=F64, device=DEV) for _ in weights]
    for c in range(0, F.shape[1], 1 << 16):
        f = F[:, c:c + (1 << 16)].double()
        for G, g in zip(out, _grams(f, [w[c:c + (1 << 16)] for w in weights])):
            G += g
    return out


def _sign(U):
    at = U.abs().argmax(1, keepdim=True)
    return U * torch.gather(U, 1, at).sign()


def _lift(Y, F, div):
    return _sign(torch.cat([(Y.T @ F[:, c:c + (1 << 18)].double()) / div[c:c + (1 << 18)]
                            for c in range(0, F.shape[1], 1 << 18)], 1))


def _eig_exact(F, d, A, C, k):
    R = torch.linalg.cholesky(A).T
    M = R @ C @ R.T
    lam, V = torch.linalg.eigh((M + M.T) / 2)
    lam, V = lam.flip(0)[:k], V.flip(1)[:, :k]
    return lam, _lift(torch.linalg.solve_triangular(R, V, upper=True), F, d)


def exact(case, seed):
    form, r, k = case["form"], case["r"], case["k"]
    if form == "factor" and case["prec"] != "fp64":
        return None     # the pivots drawn depend on the rounding of the residual diagonal
    s = prepare(case, seed)
    if form == "batch":
        out = []
        for p in _problems(case, s["seed"]):
            F, rho, piv = _pchol(p["X"], p["eps"], p["r"], "arpc", p["b"], p["seed"])
            out.append(dict(F=F, rho=rho, pivots=None))
        return out
    if form == "normalize":
        return _norm_exact(s["F"])
    if form == "eig":
        ev, U = _eig_exact(s["F"], s["d"], s["A"], s["C"], k)
        return ev, U, None
    if form == "symmetric":
        F = s["F"]
        d, _ = _degrees(F)
        As = _grams64(F, [1.0 / d])[0]
        lam, V = torch.linalg.eigh(As)
        lam, V = lam.flip(0)[:k], V.flip(1)[:, :k]
        return d, As, (lam, _lift(V / lam.sqrt(), F, d.sqrt()))
    F, rho, piv = _pchol(s["X"], s["eps"], r, case["mode"], case["b"], s["seed"])
    n = len(piv)
    out = dict(F=F, rho=rho, pivots=None, trace_err=float(rho.sum()))
    if form == "lowmem":
        W = torch.zeros(r, r, dtype=F64, device=DEV)
        W[:n, :n] = torch.tril(F[:n, piv.to(DEV)].T)
        d, q, A, C = _norm_exact(F[:n])
        A, C = (torch.nn.functional.pad(G, (0, r - n) * 2) for G in (A, C))
        return dict(W=W, rho=rho, pivots=None, trace_err=out["trace_err"], d=d, q=q, A=A, C=C)
    if form == "whole":
        d, q, A, C = _norm_exact(F[:n])
        ev, U = _eig_exact(F[:n], d, A, C, k)
        out.update(d=d, q=q, A=A, C=C, ev=ev, U=U)
    return out
