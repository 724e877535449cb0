"""Workload cases of the Kryging library, timed through its public entry points.

A case is one call that a program makes over and over: a covariance matvec, a
Gaussian-process sample, a log-determinant, a solve, a likelihood search, or
one whole likelihood-and-kriging request.  Sizes follow ``inputs.WORKLOADS``
(tiny32, grid1024, search512, the serving stream's 128..2048 sides, large4096);
``draw`` spreads over the same ranges, odd sizes included.

``exact`` recomputes a case in 64 bits with torch alone: the torus covariance
from its formula, library FFTs, conjugate gradients, fully reorthogonalised
Lanczos.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2012_13133_gb300 import kry

DEV = "cuda:0"


class _Cov:
    def __init__(self, c, nu=None, rng=None):
        self.sigma2, self.tau2 = 1.0, c["tau2"]
        self.nu = c["nu"] if nu is None else nu
        self.range = c["range"] if rng is None else rng
        self.angle, self.ratio = c.get("angle", 0.0), c.get("ratio", 1.0)


def _case(op, n1, n2, mask, missing, nu, rng, tau2, name=None, **more):
    c = dict(op=op, n1=n1, n2=n2, mask=mask, missing=missing, nu=nu, range=rng, tau2=tau2, **more)
    return c if name is None else dict(name=name, **c)


def listed():
    return [
        # the smallest grid in use (tiny32, FP64, every cell observed): one matvec, all latency
        _case("matvec", 32, 32, "full", 0.0, 0.5, 0.1, 0.1, "matvec_32_f64", prec="f64", nvec=1),
        # a small serving request's CG iteration: the [y, X] columns on a 128 x 128 grid
        _case("matvec", 128, 128, "mixed", 0.4, 0.5, 0.1, 0.1, "matvec_128_f32", prec="f32", nvec=4),
        # a ragged map tile with cloud gaps and an odd number of vectors
        _case("matvec", 363, 730, "circles", 0.35, 1.5, 0.06, 0.1, "matvec_363x730_f32", prec="f32", nvec=5),
        # grid1024: the CG batch [y, X]
        _case("matvec", 1024, 1024, "uniform", 0.5, 1.5, 0.05, 0.05, "matvec_1024_cg_f32", prec="f32", nvec=4),
        # grid1024: the Lanczos batch of 64 probes
        _case("matvec", 1024, 1024, "uniform", 0.5, 1.5, 0.05, 0.05, "matvec_1024_slq_f32", prec="f32", nvec=64),
        # large4096: the CG batch on the largest grid, anisotropic, clustered gaps
        _case("matvec", 4096, 4096, "circles", 0.3, 0.5, 0.05, 0.05, "matvec_4096_f32", prec="f32", nvec=4,
              angle=math.radians(30.0), ratio=3.0),
        # search512 in FP64: what true residuals and FP64 fits apply
        _case("matvec", 512, 512, "uniform", 0.3, 1.0, 0.08, 0.1, "matvec_512_f64", prec="f64", nvec=4),
        # one synthetic field on the grid1024 lattice (embedding eigenvalues and their use)
        _case("sample", 1024, 1024, "full", 0.0, 1.5, 0.05, 0.05, "sample_1024"),
        # log-determinant of one search512 setting: 32 probes x 50 Lanczos steps
        _case("logdet", 512, 512, "uniform", 0.3, 0.5, 0.02, 0.1, "logdet_512", nprobe=32, nsteps=50),
        # the solves K^-1 [y, X] of grid1024, to the tolerance that kry.Context.solve defaults to
        _case("solve", 1024, 1024, "uniform", 0.5, 1.5, 0.05, 0.05, "solve_1024", nrhs=4, precond=0),
        # a batched likelihood search over covariance settings
        _case("search", 256, 256, "uniform", 0.3, 0.5, 0.02, 0.1, "search_256", settings=8, nprobe=16, nsteps=50),
        # a serving request: likelihood and kriging means of a map with cloud gaps
        _case("request", 500, 437, "circles", 0.3, 0.5, 0.02, 0.1, "request_500x437", nprobe=16, nsteps=50),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choices(["matvec", "sample", "logdet", "solve", "search", "request"], [5, 1, 1, 1, 1, 1])[0]
    hi = {"matvec": 2200, "sample": 1500, "logdet": 500, "solve": 500, "search": 220, "request": 420}[op]
    lo = {"matvec": 24, "sample": 64, "logdet": 64, "solve": 64, "search": 40, "request": 64}[op]
    n1 = log_int(lo, hi)
    n2 = max(lo, min(hi, int(round(n1 * math.exp(rng.uniform(-0.7, 0.7))))))
    mask = rng.choice(["uniform", "circles", "mixed"])
    missing = round(rng.uniform(0.05, 0.6), 3)
    nu = rng.choice([0.5, 1.0, 1.5, 2.5] if op in ("matvec", "sample") else [0.5, 1.5])
    tau2 = round(rng.uniform(0.05, 0.3) if op in ("matvec", "sample") else rng.uniform(0.1, 0.2), 4)
    # the stream's ranges in domain units; the iterative calls' of 4 to 9 cells, where FP32 resolves K well
    far = rng.uniform(0.02, 0.1) if op in ("matvec", "sample") else rng.uniform(4.0, 9.0) / max(n1, n2)
    c = _case(op, n1, n2, mask, missing, nu, round(far, 4), tau2)
    if op == "matvec":
        most = max(1, min(64, (1024 * 1024 * 64) // (2 * n1 * n2)))
        c["prec"] = rng.choice(["f32", "f32", "f32", "f64"])
        c["nvec"] = log_int(1, most if c["prec"] == "f32" else max(1, min(8, most // 8)))
    elif op == "logdet":
        c["nprobe"], c["nsteps"] = rng.randint(4, 32), rng.randint(20, 60)
    elif op == "solve":
        c["nrhs"], c["precond"] = rng.randint(1, 8), rng.randint(0, 1) if mask == "circles" else 0
    elif op == "search":
        c["settings"], c["nprobe"], c["nsteps"] = rng.randint(2, 8), 2 * rng.randint(3, 8), rng.randint(30, 50)
    elif op == "request":
        c["nprobe"], c["nsteps"] = rng.randint(8, 16), rng.randint(30, 50)
    return c


# ------------------------------------------------------------------ inputs

def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + stream)
    return g


def _centres(n1, n2):
    s1 = (torch.arange(n1, device=DEV, dtype=torch.float64) + 0.5) / n1
    s2 = (torch.arange(n2, device=DEV, dtype=torch.float64) + 0.5) / n2
    return s1[:, None].expand(n1, n2), s2[None, :].expand(n1, n2)


def _mask(c, seed):
    """Observed cells: all, uniformly scattered holes, circular (cloud-like) gaps, or half of each."""
    n1, n2, N = c["n1"], c["n2"], c["n1"] * c["n2"]
    m = torch.ones(n1, n2, dtype=torch.bool, device=DEV)
    circles = {"full": 0.0, "uniform": 0.0, "circles": 1.0, "mixed": 0.5}[c["mask"]] * c["missing"]
    if circles > 0:
        s1, s2 = _centres(n1, n2)
        r = np.random.default_rng(seed)
        over = -int(round(circles * N))
        while over < 0:   # the last circle keeps as many of its cells, inmost first, as the share asks for
            a, b, q = r.random(), r.random(), r.uniform(0.02, 0.15)
            d = torch.where(m, (s1 - a) ** 2 + (s2 - b) ** 2, torch.inf).reshape(-1)
            new = torch.nonzero(d <= q * q).reshape(-1)
            new = new[torch.argsort(d[new], stable=True)][: min(new.numel(), -over)]
            m.view(-1)[new] = False
            over += new.numel()
    drop = int(round(c["missing"] * N)) - (N - int(m.sum()))
    if c["mask"] in ("uniform", "mixed") and drop > 0:
        at = torch.nonzero(m.reshape(-1)).reshape(-1)
        at = at[torch.randperm(at.numel(), device=DEV, generator=_gen(seed, 1))[: min(drop, at.numel() - 1)]]
        m.view(-1)[at] = False
    return m


def _pow2(x):
    return 1 << max(0, int(x - 1).bit_length())


def _matern(r, nu):
    x = math.sqrt(2.0 * nu) * r
    if nu == 0.5:
        return torch.exp(-x)
    if nu == 1.0:
        return torch.where(x > 0, x * torch.special.modified_bessel_k1(x.clamp_min(1e-300)), torch.ones_like(x))
    if nu == 1.5:
        return (1 + x) * torch.exp(-x)
    return (1 + x + x * x / 3) * torch.exp(-x)


def _spectrum(n1, n2, cov):
    """Eigenvalues of the torus covariance (minimal-image lags, a lag of half the torus averaging its images)."""
    M1, M2 = _pow2(2 * n1), _pow2(2 * n2)
    j1 = torch.arange(M1, device=DEV, dtype=torch.float64)
    j2 = torch.arange(M2, device=DEV, dtype=torch.float64)
    ca, sa, c = math.cos(cov.angle), math.sin(cov.angle), 0.0
    for h1 in (torch.where(2 * j1 <= M1, j1, j1 - M1), torch.where(2 * j1 < M1, j1, j1 - M1)):
        for h2 in (torch.where(2 * j2 <= M2, j2, j2 - M2), torch.where(2 * j2 < M2, j2, j2 - M2)):
            a, b = (h1 / n1)[:, None], (h2 / n2)[None, :]
            u, v = ca * a + sa * b, cov.ratio * (ca * b - sa * a)
            c = c + 0.25 * cov.sigma2 * _matern(torch.sqrt(u * u + v * v) / cov.range, cov.nu)
    return torch.fft.fft2(c.to(torch.complex128)).real


def _field(n1, n2, cov, xi):
    lam = _spectrum(n1, n2, cov).clamp_min(0.0)
    z = torch.complex(xi[0], xi[1]) * torch.sqrt(lam / lam.numel())
    return torch.fft.fft2(z).real[:n1, :n2].contiguous()


def _design(c, at):
    s1, s2 = _centres(c["n1"], c["n2"])
    s1, s2 = s1.reshape(-1)[at], s2.reshape(-1)[at]
    return torch.stack([torch.ones_like(s1), s1, s2])


def _inputs(c, seed):
    """Mask and the arrays that the case's call takes."""
    m = _mask(c, seed)
    at = torch.nonzero(m.reshape(-1)).reshape(-1)
    d = {"mask": m, "at": at}
    n1, n2, p = c["n1"], c["n2"], at.numel()
    if c["op"] == "matvec":
        d["V"] = torch.randn(c["nvec"], p, device=DEV, dtype=torch.float64, generator=_gen(seed, 2))
        d["V"] = d["V"].to(torch.float32 if c["prec"] == "f32" else torch.float64)
        return d
    if c["op"] == "logdet":
        return d
    M1, M2 = _pow2(2 * n1), _pow2(2 * n2)
    d["xi"] = torch.randn(2, M1, M2, device=DEV, dtype=torch.float64, generator=_gen(seed, 3))
    if c["op"] == "sample":
        return d
    d["X"] = _design(c, at)
    eps = torch.randn(p, device=DEV, dtype=torch.float64, generator=_gen(seed, 4))
    f = _field(n1, n2, _Cov(c), d.pop("xi"))
    beta = torch.tensor([1.0, 0.5, -0.5], device=DEV, dtype=torch.float64)
    d["y"] = (beta @ d["X"] + f.reshape(-1)[at] + math.sqrt(c["tau2"]) * eps).contiguous()
    if c["op"] == "solve":
        more = torch.randn(max(0, c["nrhs"] - 4), p, device=DEV, dtype=torch.float64, generator=_gen(seed, 5))
        d["B"] = torch.cat([d["y"][None], d["X"], more])[: c["nrhs"]].contiguous()
    if c["op"] == "request":
        d["cells"] = torch.nonzero(~m.reshape(-1)).reshape(-1)
        d["Xc"] = _design(c, d["cells"])
    return d


def _thetas(c):
    """A search's covariance settings: ranges around the case's, with the two smoothnesses of the stream."""
    return [_Cov(c, nu=(0.5, 1.5)[k % 2], rng=c["range"] * (1 + 0.25 * (k // 2))) for k in range(c["settings"])]


def _probe_seed(seed):
    return int(seed) % (1 << 20)


def prepare(case, seed):
    c, d = case, _inputs(case, seed)
    ctx = kry.Context(0)
    ctx.set_mask(d["mask"].to(torch.uint8))
    s = {"case": c, "ctx": ctx, "cov": _Cov(c), **d}
    if c["op"] in ("matvec", "logdet", "solve"):
        s["emb"] = ctx.embed(s["cov"], kry.KRY_F64 if c.get("prec") == "f64" else kry.KRY_F32)
    if c["op"] == "matvec":
        s["out"] = torch.empty_like(d["V"])
    if c["op"] == "solve":
        s["sol"] = torch.empty_like(d["B"])
    if c["op"] in ("search", "request"):
        s["opts"] = kry.Opts(prec=kry.KRY_F32, nprobe=c["nprobe"], nsteps=c["nsteps"], seed=_probe_seed(seed),
                             rtol=1e-8, maxit=20000, reorth=1, precond=2)
    s["seed"] = _probe_seed(seed)
    return s


def run(s):
    # What an FP32 run hands back in 64-bit containers (solutions, means, per-probe values) is kept
    # in FP32, the precision that was asked for.
    c, ctx = s["case"], s["ctx"]
    if c["op"] == "matvec":
        return ctx.matvec(s["emb"], s["V"], s["out"])
    if c["op"] == "sample":
        return ctx.sample(s["cov"], s["xi"].shape[1], s["xi"].shape[2], s["xi"])
    if c["op"] == "logdet":
        ld, _, per = ctx.logdet(s["emb"], c["nprobe"], c["nsteps"], s["seed"], reorth=1)
        return {"logdet": ld, "per_probe": per.astype(np.float32)}
    if c["op"] == "solve":
        x, _, _, status = ctx.solve(s["emb"], s["B"], rtol=1e-8, maxit=20000, X=s["sol"], precond=bool(c["precond"]))
        return {"x": x.float(), "status": status}
    if c["op"] == "search":
        r = ctx.profile_loglik(s["y"], s["X"], _thetas(c), s["opts"])
        return {"loglik": r["loglik"].astype(np.float32), "logdet": r["logdet"].astype(np.float32),
                "beta": r["beta"].astype(np.float32), "status": r["status"]}
    r = ctx.loglik_krige(s["cov"], s["opts"], s["y"], s["X"], cells=s["cells"], Xc=s["Xc"])
    return {"loglik": r["loglik"], "logdet": r["logdet"], "beta": r["beta"].astype(np.float32),
            "mean": r["mean_cells"].float(), "status": r["status"]}


def work(case):
    """Bytes of the inputs and results of one pass, and the arithmetic of its FFTs (5 L log2 L each)."""
    c = case
    n1, n2 = c["n1"], c["n2"]
    p = (1.0 - c["missing"]) * n1 * n2
    fft = 2 * n1 * 10.0 * n2 * math.log2(2 * n2) + 4 * n2 * 10.0 * n1 * math.log2(2 * n1)   # one complex pair, both ways
    if c["op"] == "matvec":
        w = 8 if c["prec"] == "f64" else 4
        return {"bytes": 2 * w * c["nvec"] * p + w * n1 * n2 + 4 * p, "flops": fft * c["nvec"] / 2}
    if c["op"] == "sample":
        return {"bytes": 8.0 * (2 * _pow2(2 * n1) * _pow2(2 * n2) + n1 * n2), "flops": 2 * fft}
    if c["op"] == "logdet":
        return {"bytes": 4.0 * p, "flops": fft * c["nprobe"] * c["nsteps"] / 2}
    if c["op"] == "solve":   # an iteration count of a few hundred is what such a system takes
        return {"bytes": 8.0 * c["nrhs"] * 2 * p, "flops": 300 * fft * c["nrhs"] / 2}
    k = c.get("settings", 1)
    return {"bytes": 8.0 * (4 * p + (4 * (n1 * n2 - p) if c["op"] == "request" else 0)),
            "flops": k * fft * (c["nprobe"] * c["nsteps"] / 2 + 2 * 200)}


# ------------------------------------------------------------------ 64-bit results

class _K64:
    """K = A Sigma A^T + tau2 I on the observed cells, by library FFTs in 64 bits."""

    def __init__(self, n1, n2, at, cov):
        self.n1, self.n2, self.at, self.tau2 = n1, n2, at, cov.tau2
        self.lam = _spectrum(n1, n2, cov)

    def grid(self, v):
        """Sigma A^T v on every cell, rows of v in pairs."""
        n1, n2 = self.n1, self.n2
        out = torch.empty(v.shape[0], n1 * n2, device=DEV, dtype=torch.float64)
        for k in range(0, v.shape[0], 2):
            z = torch.zeros(n1 * n2, device=DEV, dtype=torch.complex128)
            z[self.at] = torch.complex(v[k], v[k + 1] if k + 1 < v.shape[0] else torch.zeros_like(v[k]))
            z = torch.fft.ifft2(self.lam * torch.fft.fft2(z.view(n1, n2), s=self.lam.shape))[:n1, :n2].reshape(-1)
            out[k] = z.real
            if k + 1 < v.shape[0]:
                out[k + 1] = z.imag
        return out

    def __call__(self, v):
        return self.grid(v)[:, self.at] + self.tau2 * v

    def solve(self, b, tol=1e-12, maxit=6000):
        x, r = torch.zeros_like(b), b.clone()
        q, rr = r.clone(), (r * r).sum(1)
        goal = tol * tol * rr
        for it in range(maxit):
            kq = self(q)
            a = rr / (q * kq).sum(1).clamp_min(1e-300)
            x += a[:, None] * q
            r -= a[:, None] * kq
            new = (r * r).sum(1)
            if it % 16 == 15 and bool((new <= goal).all()):
                break
            q = r + (new / rr.clamp_min(1e-300))[:, None] * q
            rr = new
        return x

    def quadrature(self, nprobe, nsteps, seed):
        """z^T log(K) z by Lanczos quadrature with a fully reorthogonalised basis, for the library's probes."""
        p = self.at.numel()
        i = torch.arange(p, device=DEV, dtype=torch.int64)
        z = torch.stack([_rademacher(seed ^ (k << 32), i) for k in range(nprobe)])
        q = z / math.sqrt(p)
        Q, al, be = [q], [], []
        for j in range(nsteps):
            w = self(Q[j])
            a = (w * Q[j]).sum(1)
            al.append(a)
            if j + 1 == nsteps:
                break
            w = w - a[:, None] * Q[j] - (be[-1][:, None] * Q[j - 1] if j else 0.0)
            for _ in range(2):
                for u in Q:
                    w = w - (w * u).sum(1)[:, None] * u
            b = torch.linalg.vector_norm(w, dim=1)
            be.append(b)
            Q.append(w / b[:, None])
        T = torch.diag_embed(torch.stack(al, 1))
        if be:
            o = torch.stack(be, 1)
            T = T + torch.diag_embed(o, 1) + torch.diag_embed(o, -1)
        t, U = torch.linalg.eigh(T.cpu())
        return p * (U[:, 0, :] ** 2 * torch.log(t.clamp_min(self.tau2))).sum(1)


def _rademacher(key, i):
    """+1 where the top bit of splitmix64(key xor i) is 0, else -1."""
    def shr(x, n):
        return (x >> n) & ((1 << (64 - n)) - 1)

    x = (i ^ key) + (0x9E3779B97F4A7C15 - (1 << 64))
    x = (x ^ shr(x, 30)) * (0xBF58476D1CE4E5B9 - (1 << 64))
    x = (x ^ shr(x, 27)) * (0x94D049BB133111EB - (1 << 64))
    return torch.where((x ^ shr(x, 31)) < 0, -1.0, 1.0).to(torch.float64)


def _gls(K, d, ld):
    V = torch.cat([d["y"][None], d["X"]])
    Z = K.solve(V)
    G = V @ Z.T
    beta = torch.linalg.solve(G[1:, 1:], G[1:, 0])
    quad = G[0, 0] - beta @ G[1:, 0]
    ll = -0.5 * (ld + quad + d["y"].numel() * math.log(2 * math.pi))
    return float(ll), beta, Z[0] - beta @ Z[1:]


def exact(case, seed):
    c = case
    n1, n2, cov = c["n1"], c["n2"], _Cov(case)
    # iterative cases on large grids take minutes in 64 bits
    if c["op"] in ("logdet", "solve", "search", "request") and n1 * n2 > 300_000:
        return None
    d = _inputs(c, seed)
    if c["op"] == "sample":
        return _field(n1, n2, cov, d["xi"])
    if c["op"] == "matvec":
        return _K64(n1, n2, d["at"], cov)(d["V"].double())
    if c["op"] == "solve":
        return {"x": _K64(n1, n2, d["at"], cov).solve(d["B"]), "status": None}
    if c["op"] == "logdet":
        per = _K64(n1, n2, d["at"], cov).quadrature(c["nprobe"], c["nsteps"], _probe_seed(seed))
        return {"logdet": float(per.mean()), "per_probe": per}
    if c["op"] == "search":
        ll, lds, betas = [], [], []
        for th in _thetas(c):
            K = _K64(n1, n2, d["at"], th)
            ld = float(K.quadrature(c["nprobe"], c["nsteps"], _probe_seed(seed)).mean())
            v, beta, _ = _gls(K, d, ld)
            ll.append(v), lds.append(ld), betas.append(beta.cpu().numpy())
        return {"loglik": np.array(ll), "logdet": np.array(lds), "beta": np.array(betas), "status": None}
    K = _K64(n1, n2, d["at"], cov)
    ld = float(K.quadrature(c["nprobe"], c["nsteps"], _probe_seed(seed)).mean())
    ll, beta, w = _gls(K, d, ld)
    mean = K.grid(w[None])[0][d["cells"]] + beta @ d["Xc"]
    return {"loglik": ll, "logdet": ld, "beta": beta, "mean": mean, "status": None}
