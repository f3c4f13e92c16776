"""Performance cases of the FIFA-GP library: what users run, through the public binding.

Every case is a dict of plain values; ``kind`` names the entry points it goes through:

* ``loglik``   fifa_assemble, fifa_shift_scale, fifa_factor, fifa_logdet, fifa_solve: one evaluation of the marginal
               likelihood's log-determinant and (s C~ + I)^-1 y at a length-scale (what a hyperparameter search calls);
* ``gibbs``    fifa_gibbs_step(1) and fifa_chain_get: one iteration of the sampler, with its state read back;
* ``sample``   fifa_sample: one Algorithm 1 draw and posterior mean with factors that are kept;
* ``matvec``   fifa_matvec: products with two vectors;
* ``predict``  fifa_predict: posterior mean and variance at new inputs, inside and beyond the data;
* ``hetero``   fifa_add_diagonal, fifa_factor, fifa_sample_hetero: Algorithm 1.h with per-point noise that changes;
* ``additive`` fifa_additive_sweep(1): one block-Gibbs sweep of the d-dimensional additive model;
* ``serving``  fifa_server_submit / fifa_server_wait: a burst of small and mid-size requests, host data in and out.

Inputs follow the repository's workloads (paper_2006_06537_gb300/inputs.py): sorted uniform points, or eight narrow
clusters, with a noisy sum of sinusoids.  The nugget grows with n beyond 8192 so that C~'s condition number, and with it
how well the draws are determined, does not.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2006_06537_gb300 import fifa

CAP = 32  # ACA rank cap of every workload in this repository


def listed():
    return [
        # the smallest call: a likelihood evaluation for a few hundred points (latency and launches)
        dict(name="loglik_500", kind="loglik", n=500, data="uniform", kernel="se", rho=0.1, leaf=32, eps=1e-12, prec="fp64"),
        # a hyperparameter search on an odd-sized large set: assembly and factorization
        dict(name="loglik_300007", kind="loglik", n=300007, data="clustered", kernel="se", rho=0.01, leaf=32, eps=1e-10, prec="fp64"),
        # the small sampler: n = 2048, SE, leaf 64, tolerance 1e-12, FP64
        dict(name="gibbs_2048", kind="gibbs", n=2048, data="uniform", kernel="se", rho=0.1, leaf=64, eps=1e-12, prec="fp64"),
        # the Matern-5/2 sampler: n = 131072, leaf 128, FP64
        dict(name="gibbs_131072", kind="gibbs", n=131072, data="uniform", kernel="matern", rho=0.05, leaf=128, eps=1e-10, prec="fp64"),
        # the benchmark's sampler: n = 2^20 in clusters, SE, leaf 32, mixed precision
        dict(name="gibbs_1048576", kind="gibbs", n=1048576, data="clustered", kernel="se", rho=0.01, leaf=32, eps=1e-10, prec="mixed"),
        # repeated draws at fixed hyperparameters, mid size, mixed precision (conjugate gradients, FP32 preconditioner)
        dict(name="sample_65537", kind="sample", n=65537, data="uniform", kernel="se", rho=0.1, leaf=32, eps=1e-10, prec="mixed"),
        # products with the largest H-matrix (an iterative method of the user's own), an odd size
        dict(name="matvec_1000003", kind="matvec", n=1000003, data="clustered", kernel="se", rho=0.01, leaf=32, eps=1e-10, prec="fp64"),
        # posterior mean and variance at a few hundred new inputs
        dict(name="predict_10000", kind="predict", n=10000, m=301, data="uniform", kernel="matern", rho=0.05, leaf=64, eps=1e-10, prec="fp64"),
        # per-point noise re-estimated by the caller between draws
        dict(name="hetero_20011", kind="hetero", n=20011, data="uniform", kernel="matern", rho=0.05, leaf=64, eps=1e-10, prec="fp64"),
        # the additive model of the benchmark: d = 4, n = 65536, mixed precision
        dict(name="additive_65536", kind="additive", n=65536, d=4, kernel="se", rho=0.1, leaf=32, eps=1e-10, prec="mixed"),
        # a burst of requests of the serving workload's kinds, log-uniform sizes
        dict(name="serving_12", kind="serving", count=12, nmin=1024, nmax=32768, iters=8, leaf=32, eps=1e-10, prec="mixed"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["loglik", "loglik", "gibbs", "gibbs", "sample", "matvec", "predict", "hetero", "additive", "serving"])
    leaf, eps = rng.choice([32, 32, 64, 128]), rng.choice([1e-10, 1e-10, 1e-12])
    if kind == "serving":
        return dict(kind=kind, count=rng.randint(4, 12), nmin=1024, nmax=_log_int(rng, 4096, 32768), iters=rng.randint(4, 8),
                    leaf=32, eps=1e-10, prec=rng.choice(["mixed", "fp64"]))
    kernel = rng.choice(["se", "se", "matern"])
    if kind == "additive":
        return dict(kind=kind, n=_log_int(rng, 2000, 65536), d=rng.randint(2, 4), kernel=kernel, rho=round(rng.uniform(0.05, 0.15), 4),
                    leaf=32, eps=1e-10, prec=rng.choice(["mixed", "fp64"]))
    lo, hi = {"loglik": (300, 300000), "gibbs": (1000, 1000000), "sample": (2000, 500000), "matvec": (2000, 1000000),
              "predict": (1000, 40000), "hetero": (1000, 100000)}[kind]
    n = _log_int(rng, lo, hi)
    data = rng.choice(["uniform", "clustered"]) if n >= 4000 else "uniform"
    if n > 200000:
        data, kernel, leaf, eps = "clustered", "se", 32, 1e-10  # the benchmark's recipe: what runs at this size
    rho = round(rng.uniform(0.01, 0.015) if data == "clustered" else rng.uniform(0.05, 0.12), 4)
    prec = rng.choice(["fp64", "mixed"]) if kind in ("gibbs", "sample", "loglik") else "fp64"
    case = dict(kind=kind, n=n, data=data, kernel=kernel, rho=rho, leaf=leaf, eps=eps, prec=prec)
    if kind == "predict":
        case["m"] = rng.randint(100, 301)
    return case


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
TAU2, NOISE = 1.0, 0.1  # the state a running chain is in: unit signal variance, the data's noise
SIGMA2 = NOISE * NOISE


def _nugget(n):
    return 1e-6 * max(1.0, n / 8192.0)


def _points(n, data, g):
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    if data == "clustered":
        c = torch.randint(0, 8, (n,), generator=g, device="cuda")
        u = (2.0 * c + 1.0) / 16.0 + 0.02 * (u - 0.5)
    return u


def _signal(x, g, terms=4):
    a = torch.randn(terms, generator=g, device="cuda", dtype=torch.float64)
    ph = 2 * math.pi * torch.rand(terms, generator=g, device="cuda", dtype=torch.float64)
    y = torch.zeros_like(x)
    for k in range(terms):
        y += (0.5 + a[k].abs()) / (k + 1) * torch.sin(2 * math.pi * (k + 1) * x + ph[k])
    return y / y.std()


def _data(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = _points(case["n"], case["data"], g).sort().values.contiguous()
    y = _signal(x, g) + NOISE * torch.randn(x.shape, generator=g, device="cuda", dtype=torch.float64)
    return g, x, y.contiguous()


def _kernel(case):
    return fifa.FIFA_KERNEL_SE if case["kernel"] == "se" else fifa.FIFA_KERNEL_MATERN52


def _hyper(case, n):
    return fifa.fifa_hyper(_kernel(case), TAU2, case["rho"], SIGMA2, _nugget(n))


def _prior(rho):
    return fifa.fifa_prior(1.0, 1.0, 1.0, 1.0, math.log(rho), 1.0, 0.2)


def _opts(case, overlap=1):
    return fifa.fifa_opts(case["leaf"], case["eps"], CAP, fifa.FIFA_MIXED if case["prec"] == "mixed" else fifa.FIFA_FP64,
                          1e-12, 8, 0, 0, 0, overlap)


class _State:
    """A context on its own stream, with what it holds; everything is released with it."""

    def __init__(self, case, blocks=1):
        self.case = case
        self.stream = torch.cuda.Stream()
        self.stream.wait_stream(torch.cuda.current_stream())
        o = _opts(case)
        nbytes = int(1.05 * blocks * fifa.fifa_chain_bytes(o, case["n"])) + (64 << 20)
        self.ctx = fifa.Context(leaf_size=o.leaf_size, aca_tol=o.aca_tol, rank_cap=o.rank_cap, prec=o.prec,
                                refine_tol=o.refine_tol, refine_max=o.refine_max, arena_bytes=nbytes, stream=self.stream,
                                overlap_proposal=o.overlap_proposal)
        self.h = self.ctx.h
        self.objects = []  # (destructor, handle), released last to first

    def keep(self, destroy, handle):
        self.objects.append((destroy, handle))
        return handle

    def __del__(self):
        for destroy, handle in reversed(getattr(self, "objects", [])):
            destroy(self.h, handle)
        if hasattr(self, "ctx"):
            self.ctx.close()


class _Server:
    def __init__(self, case, seed):
        self.case = case
        r = np.random.default_rng(seed)
        sizes = np.exp(np.linspace(math.log(case["nmin"]), math.log(case["nmax"]), case["count"]))
        self.requests = []
        for i, n in enumerate(int(v) for v in sizes):
            x = np.sort(r.uniform(0.0, 1.0, n))
            y = NOISE * r.standard_normal(n)
            for k in range(1, 5):
                y += r.standard_normal() / k * np.sin(2 * math.pi * r.integers(1, 9) * x + r.uniform(0, 2 * math.pi))
            rho = 0.1 if i % 2 == 0 else 0.05
            init = fifa.fifa_hyper(i % 2, TAU2, rho, SIGMA2, _nugget(n))
            self.requests.append((x, y, init, _prior(rho), int(r.integers(1 << 40))))
        o = _opts(case)
        budget = int(1.1 * sum(fifa.fifa_chain_bytes(o, len(q[0])) for q in self.requests)) + (256 << 20)
        # eight workers, two of them wide: the benchmark's shares of its twenty and four
        self.handle = fifa.fifa_server_create(o, budget, 8, 1 << 13, 2)

    def __del__(self):
        if hasattr(self, "handle"):
            fifa.fifa_server_destroy(self.handle)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serving":
        return _Server(case, seed)
    n = case["n"]
    if kind == "additive":
        g = torch.Generator(device="cuda").manual_seed(seed)
        X = torch.rand((case["d"], n), generator=g, device="cuda", dtype=torch.float64)
        y = NOISE * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
        for k in range(case["d"]):
            y += _signal(X[k], g, 2)
        s = _State(case, blocks=case["d"])
        s.F = torch.empty_like(X)
        s.model = s.keep(fifa.fifa_destroy_additive,
                         fifa.fifa_additive_create(s.h, X, y, n, case["d"], _hyper(case, n), _prior(case["rho"]), seed))
        return s
    g, x, y = _data(case, seed)
    s = _State(case)
    s.x, s.y, s.seed = x, y, seed
    s.f, s.mean = torch.empty_like(y), torch.empty_like(y)
    hyper = _hyper(case, n)
    if kind == "loglik":
        s.out = torch.empty_like(y)
        return s
    if kind == "gibbs":
        s.chain = s.keep(fifa.fifa_destroy_chain,
                         fifa.fifa_chain_create(s.h, x, y, n, hyper, _prior(case["rho"]), seed, 0))
        return s
    s.C = s.keep(fifa.fifa_destroy_hmat, fifa.fifa_assemble(s.h, x, n, hyper))
    if kind == "matvec":
        s.v = torch.randn((2, n), generator=g, device="cuda", dtype=torch.float64)
        s.out = torch.empty_like(s.v)
        s.stream.wait_stream(torch.cuda.current_stream())
        return s
    s.WC = s.keep(fifa.fifa_destroy_fact, fifa.fifa_factor(s.h, s.C))
    if kind == "sample":
        M = s.keep(fifa.fifa_destroy_hmat, fifa.fifa_shift_scale(s.h, s.C, TAU2 / SIGMA2))
        s.WM = s.keep(fifa.fifa_destroy_fact, fifa.fifa_factor(s.h, M))
    elif kind == "predict":
        s.fin = _signal(x, g)
        lo, hi = x[0] - 2 * case["rho"], x[-1] + 2 * case["rho"]
        s.xs = lo + (hi - lo) * torch.rand(case["m"], generator=g, device="cuda", dtype=torch.float64)
        s.mu, s.var = torch.empty_like(s.xs), torch.empty_like(s.xs)
    elif kind == "hetero":
        s.d = torch.exp(torch.randn(n, generator=g, device="cuda", dtype=torch.float64) * 0.5) / SIGMA2
        s.dinv = 1.0 / s.d
    s.stream.wait_stream(torch.cuda.current_stream())
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "serving":
        ids = [fifa.fifa_server_submit(s.handle, x, y, init, prior, seed, i, case["iters"], case["iters"] // 2, 2)
               for i, (x, y, init, prior, seed) in enumerate(s.requests)]
        out = []
        for rid, q in zip(ids, s.requests):
            mean, draws = np.empty(len(q[0])), np.empty((2, len(q[0])))
            fifa.fifa_server_wait(s.handle, rid, mean, draws)
            out.append((mean, draws))
        return out
    n = case["n"]
    if kind == "loglik":
        C = fifa.fifa_assemble(s.h, s.x, n, _hyper(case, n))
        M = fifa.fifa_shift_scale(s.h, C, TAU2 / SIGMA2)
        W = fifa.fifa_factor(s.h, M)
        fifa.fifa_solve(s.h, W, s.y, s.out, 1)
        logdet, _ = fifa.fifa_logdet(s.h, W)
        fifa.fifa_destroy_fact(s.h, W)
        fifa.fifa_destroy_hmat(s.h, M)
        fifa.fifa_destroy_hmat(s.h, C)
        return {"logdet": logdet, "x": s.out}
    if kind == "gibbs":
        fifa.fifa_gibbs_step(s.h, s.chain, 1)
        h = fifa.fifa_chain_get(s.h, s.chain, s.f, s.mean)
        return {"f": s.f, "mean": s.mean, "sigma2": h.sigma2, "tau2": h.tau2, "rho": h.rho}
    if kind == "sample":
        fifa.fifa_sample(s.h, s.C, s.WC, s.WM, s.y, TAU2, SIGMA2, s.seed, 0, 0, s.f, s.mean)
        return {"f": s.f, "mean": s.mean}
    if kind == "matvec":
        fifa.fifa_matvec(s.h, s.C, s.v, s.out, 2)
        return {"y": s.out}
    if kind == "predict":
        fifa.fifa_predict(s.h, s.C, s.WC, s.x, s.fin, s.xs, case["m"], TAU2, s.mu, s.var)
        return {"mu": s.mu, "var": s.var}
    if kind == "hetero":
        P = fifa.fifa_add_diagonal(s.h, s.C, TAU2, s.dinv)
        WP = fifa.fifa_factor(s.h, P)
        fifa.fifa_sample_hetero(s.h, s.C, s.WC, WP, s.y, TAU2, s.d, s.seed, 0, 0, s.f, s.mean)
        fifa.fifa_destroy_fact(s.h, WP)
        fifa.fifa_destroy_hmat(s.h, P)
        return {"f": s.f, "mean": s.mean}
    fifa.fifa_additive_sweep(s.h, s.model, 1)
    sigma2, blocks = fifa.fifa_additive_get(s.h, s.model, case["d"], s.F)
    return {"F": s.F, "sigma2": sigma2, "tau2": [b.tau2 for b in blocks], "rho": [b.rho for b in blocks]}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Vectors in and out once, and the dense leaves' arithmetic: entries of the leaves (16 operations each where they
    are evaluated), their Cholesky factors and triangular solves, products with them; per tree level one off-diagonal
    basis of rank 4 per side."""
    kind = case["kind"]
    if kind == "serving":
        sizes = np.exp(np.linspace(math.log(case["nmin"]), math.log(case["nmax"]), case["count"]))
        one = [work(dict(case, kind="gibbs", n=int(n))) for n in sizes]
        return {"bytes": sum(16 * int(n) + 24 * int(n) for n in sizes), "flops": case["iters"] * sum(w["flops"] for w in one)}
    n, B = case["n"], case["leaf"]
    L = max(0, math.ceil(math.log2(max(1.0, n / B))))
    entries = n * B / 2 + 2 * 5 * n * L          # kernel entries of the leaves and of rank-4 cross approximations
    assemble = 16 * entries
    factor = n * B * B / 3 + 2 * 4 * 4 * n * L   # leaf Cholesky; one rank-4 basis per row and level
    apply_ = 2 * n * B + 4 * 4 * n * L           # a product or a solve with one vector
    matrix = 8 * (n * B / 2 + 4 * n * L)         # an H-matrix or factor that is kept, read once
    if kind == "loglik":
        return {"bytes": 24 * n, "flops": assemble + factor + 2 * apply_}
    if kind == "gibbs":
        return {"bytes": 40 * n, "flops": assemble + 2 * factor + 8 * apply_}
    if kind == "sample":
        return {"bytes": 24 * n + 3 * matrix, "flops": 6 * apply_}
    if kind == "matvec":
        return {"bytes": 32 * n + matrix, "flops": 2 * apply_}
    if kind == "predict":
        return {"bytes": 16 * n + 24 * case["m"] + matrix, "flops": (case["m"] + 2) * apply_ + 32 * n * case["m"]}
    if kind == "hetero":
        return {"bytes": 40 * n + 2 * matrix, "flops": factor + 6 * apply_}
    return {"bytes": 8 * n * (2 * case["d"] + 1), "flops": case["d"] * (assemble + 2 * factor + 8 * apply_)}


# ---------------------------------------------------------------------------
# The same in 64 bits, without the library
# ---------------------------------------------------------------------------
def _k(case, a, b):
    d = (a[:, None] - b[None, :]).abs()
    if case["kernel"] == "se":
        return torch.exp(-0.5 * (d / case["rho"]) ** 2)
    t = math.sqrt(5.0) * d / case["rho"]
    return (1 + t + t * t / 3) * torch.exp(-t)


def exact(case, seed):
    """Dense linear algebra where the size allows it (n up to 12000; products up to 2e11 kernel entries)."""
    kind = case["kind"]
    if kind in ("serving", "additive"):
        return None  # draws from the library's own random streams
    n = case["n"]
    if kind == "matvec":
        span = n * n / 8 if case["data"] == "clustered" else n * n  # points of other clusters are 10 rho away
        if span > 2e11:
            return None
        g, x, y = _data(case, seed)
        v = torch.randn((2, n), generator=g, device="cuda", dtype=torch.float64)
        out = _nugget(n) * v
        reach = 6.0 * math.sqrt(2.0) * case["rho"] if case["kernel"] == "se" else 20.0 * case["rho"]
        step = max(1, int(2e8) // n)
        for a in range(0, n, step):
            xa = x[a:a + step]
            lo = int(torch.searchsorted(x, xa[0] - reach)) if case["data"] == "clustered" else 0
            hi = int(torch.searchsorted(x, xa[-1] + reach)) if case["data"] == "clustered" else n
            out[:, a:a + step] += (_k(case, xa, x[lo:hi]) @ v[:, lo:hi].T).T
        return {"y": out}
    if n > 12000:
        return None
    g, x, y = _data(case, seed)
    eye = torch.eye(n, device="cuda", dtype=torch.float64)
    C = _k(case, x, x) + _nugget(n) * eye
    if kind == "predict":
        fin = _signal(x, g)
        lo, hi = x[0] - 2 * case["rho"], x[-1] + 2 * case["rho"]
        xs = lo + (hi - lo) * torch.rand(case["m"], generator=g, device="cuda", dtype=torch.float64)
        W = torch.linalg.cholesky(C)
        c = _k(case, x, xs)
        z = torch.linalg.solve_triangular(W, c, upper=False)
        zf = torch.linalg.solve_triangular(W, fin[:, None], upper=False)
        return {"mu": (z.T @ zf)[:, 0], "var": TAU2 * (1.0 - (z * z).sum(0))}
    if kind == "hetero":
        d = torch.exp(torch.randn(n, generator=g, device="cuda", dtype=torch.float64) * 0.5) / SIGMA2
        r = torch.linalg.solve(TAU2 * C + torch.diag(1.0 / d), y)
        return {"f": None, "mean": TAU2 * (C @ r)}
    W = torch.linalg.cholesky(TAU2 / SIGMA2 * C + eye)
    r = torch.cholesky_solve(y[:, None], W)[:, 0]
    if kind == "loglik":
        return {"logdet": float(2 * W.diagonal().log().sum()), "x": r}
    mean = TAU2 / SIGMA2 * (C @ r)
    if kind == "sample":
        return {"f": None, "mean": mean}
    return {"f": None, "mean": mean, "sigma2": None, "tau2": None, "rho": None}
