"""The measured cases: the calls a user of the library makes, at the sizes of its own workloads.

A case is a dict of plain values.  Kinds:
  plain       one Gibbs chain on the whole matrix: restart, n sweeps, posterior means
  pp          a posterior-propagation run on an I x J grid: restart, three stages, aggregated means
  grad        the log-joint and its gradients through the autograd function (forward + backward)
  langevin    unadjusted Langevin moves on caller-owned FP32 factors
  summaries   lambda-means clustering and mixture fits of retained samples (bmf_fit_summaries)
  aggregate   Eq. 14 / Algorithm 2 on device arrays without allocation (bmf_aggregate_static)

Chains draw from the device generator unless a case says otherwise, and keep the default launch
schedule except where a case names the graph launch.  In the reduced-precision modes (fp32,
bf16, tf32 gathers) the posterior means are handed on as float32, which is what these modes
carry; the FP64 mode's stay float64."""
from __future__ import annotations

import math

import numpy as np
import torch

DEV = "cuda"
F64 = torch.float64


# ------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------
def listed():
    return [
        # a first look at a small matrix (the planted parity workload): launches and latency
        dict(name="planted-k10-fp64", kind="plain", N=1000, D=500, M=25_000, pattern="uniform", K=10,
             prec="fp64", sweeps=10, burnin=2, sigma=0.5, ratings=False, noise="fixed"),
        # MovieLens-shaped ratings, the plain FP32 sampler with its per-sweep test monitor
        dict(name="zipf10M-k10-fp32", kind="plain", N=69_878, D=10_677, M=10_000_000, pattern="zipf1.2",
             K=10, prec="fp32", sweeps=100, burnin=20, sigma=0.8, ratings=True, noise="fixed"),
        # the same data in the full FP64 mode (the default precision)
        dict(name="zipf10M-k10-fp64", kind="plain", N=69_878, D=10_677, M=10_000_000, pattern="zipf1.2",
             K=10, prec="fp64", sweeps=20, burnin=4, sigma=0.8, ratings=True, noise="fixed"),
        # the paper's simulated data on a 10 x 10 grid, FP64 as in the partition experiment:
        # many small subsets, launched as one CUDA graph per stage
        dict(name="sim-pp10x10-k5-fp64", kind="pp", N=6040, D=3706, M=4_476_848, pattern="uniform", K=5,
             prec="fp64", I=10, J=10, sweeps=200, burnin=100, thin=2, sigma=1.0, graph=1),
        # the posterior-propagation benchmark workload: stages of 1 / 6 / 9 uneven subsets
        dict(name="pp4x4-k16-fp32", kind="pp", N=100_000, D=20_000, M=20_000_000, pattern="zipf1.2", K=16,
             prec="fp32", I=4, J=4, sweeps=120, burnin=40, thin=1, sigma=0.5, graph=0),
        # the K = 32 ratings workload at a quarter of its rows and columns, BF16 gathers
        dict(name="zipf6M-k32-bf16", kind="plain", N=120_047, D=4_442, M=6_250_000, pattern="zipf1.1",
             K=32, prec="bf16", sweeps=20, burnin=4, sigma=0.8, ratings=True, noise="fixed"),
        # an odd size with a noise precision sampled per column, single-pass TF32
        dict(name="zipf1M-k24-tf32-noise", kind="plain", N=30_011, D=2_027, M=1_000_003, pattern="zipf1.2",
             K=24, prec="tf32", sweeps=20, burnin=4, sigma=0.5, ratings=False, noise="column"),
        # the widest latent dimension: Gibbs sweeps of the K = 64 workload at a quarter size
        dict(name="uniform3M-k64-fp32", kind="plain", N=50_000, D=12_500, M=3_125_000, pattern="uniform",
             K=64, prec="fp32", sweeps=10, burnin=2, sigma=0.3, ratings=False, noise="fixed"),
        # gradients of the log-joint at K = 64 (half size), forward and backward
        dict(name="grad12M-k64", kind="grad", N=100_000, D=25_000, M=12_500_000, pattern="uniform", K=64,
             sigma=0.3),
        # Langevin moves beside the sampler on rating data
        dict(name="langevin2M-k10", kind="langevin", N=34_939, D=5_338, M=2_500_000, pattern="zipf1.2", K=10,
             sigma=0.8, steps=10),
        # mixture summaries of 200 retained samples per row (the paper's PP GMM setting)
        dict(name="gmm-20000x200-k10", kind="summaries", R=20_000, S=200, K=10, C=3, modes=3),
        # submodel aggregation by a caller that owns all device memory, near the call's row limit
        dict(name="aggregate-40000x4-k10", kind="aggregate", R=40_000, J=4, K=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plain", "plain", "plain", "pp", "pp", "grad", "langevin", "summaries", "aggregate"])
    pattern = rng.choice(["uniform", "zipf1.1", "zipf1.2"])
    if kind == "summaries":
        K = rng.randint(2, 16)
        return dict(kind=kind, R=_log(rng, 500, 20_000), S=rng.randint(60, 200), K=K, C=rng.randint(1, 4),
                    modes=rng.randint(1, 3))
    if kind == "aggregate":
        K = rng.randint(3, 16)
        return dict(kind=kind, R=_log(rng, 500, 4_000_000 // (K * K)), J=rng.randint(2, 6), K=K)
    if kind in ("grad", "langevin"):
        N = _log(rng, 3_000, 100_000)
        D = max(200, N // rng.randint(2, 9))
        c = dict(kind=kind, N=N, D=D, M=N * rng.randint(15, 60), pattern=pattern, K=rng.randint(2, 64),
                 sigma=0.5)
        return dict(c, steps=rng.randint(2, 10)) if kind == "langevin" else c
    N = _log(rng, 900, 70_000)
    D = max(150, N // rng.randint(2, 12))
    M = min(N * rng.randint(12, 120), N * D // 8)
    if kind == "pp":
        K = rng.randint(3, 18)
        return dict(kind=kind, N=N, D=D, M=M, pattern=pattern, K=K, prec=rng.choice(["fp64", "fp32", "fp32"]),
                    I=rng.randint(1, 5), J=rng.randint(2, 5), sweeps=100, burnin=20, thin=1, sigma=0.5,
                    graph=rng.randint(0, 1))
    K = rng.randint(1, 16) if rng.random() < 0.6 else rng.randint(17, 64)
    prec = rng.choice(["fp64", "fp32", "fp32", "bf16", "tf32"])
    if prec == "fp64" and K > 16:
        M = min(M, 1_000_000)
    return dict(kind=kind, N=N, D=D, M=M, pattern=pattern, K=K, prec=prec, sweeps=rng.randint(5, 20), burnin=2,
                sigma=0.5, ratings=False, noise=rng.choice(["fixed", "fixed", "fixed", "column"]))


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
def _gen(seed, part):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1_000_003 + part) & 0x7FFFFFFFFFFFFFFF)


def _pairs(c, seed):
    """M distinct (row, col) pairs: uniform, or the product model with Zipf weights over randomly
    permuted ranks (a heavy row and column meet in almost every cell)."""
    N, D, M = c["N"], c["D"], min(c["M"], c["N"] * c["D"] // 2)
    g = _gen(seed, 1)
    if c["pattern"] == "uniform":
        def some(m):
            return torch.randint(0, N * D, (m,), generator=g, device=DEV)
    else:
        s = float(c["pattern"][4:])

        def cdf(n):
            w = (torch.randperm(n, generator=g, device=DEV) + 1).to(F64) ** -s
            return torch.cumsum(w / w.sum(), 0)
        p, q = cdf(N), cdf(D)

        def some(m):
            u = torch.rand(2, m, generator=g, device=DEV, dtype=F64)
            r = torch.searchsorted(p, u[0]).clamp_(max=N - 1)
            return r * D + torch.searchsorted(q, u[1]).clamp_(max=D - 1)
    keys = torch.unique(some(M + M // 8 + 1024))
    while keys.numel() < M:
        keys = torch.unique(torch.cat([keys, some(2 * M)]))
    keys = keys[torch.randperm(keys.numel(), generator=g, device=DEV)[:M]]
    return torch.div(keys, D, rounding_mode="floor"), keys % D


def _matrix(c, seed):
    """Training and held-out (10%) entries with values of a rank-K truth, and initial states."""
    N, D, K = c["N"], c["D"], c["K"]
    r, q = _pairs(c, seed)
    g = _gen(seed, 2)
    sd = K ** -0.25 if c.get("ratings") else 1.0
    X = torch.randn(N, K, generator=g, device=DEV) * sd
    W = torch.randn(D, K, generator=g, device=DEV) * sd
    y = torch.empty(r.numel(), device=DEV)
    for a in range(0, r.numel(), 1 << 21):
        y[a:a + (1 << 21)] = (X[r[a:a + (1 << 21)]] * W[q[a:a + (1 << 21)]]).sum(1)
    y = (y + torch.randn(y.numel(), generator=g, device=DEV) * c["sigma"]).to(F64)
    if c.get("ratings"):
        y = (3.5 + y).round().clamp(1.0, 5.0)
    nt = r.numel() // 10
    r, q = r.to(torch.int32), q.to(torch.int32)
    X0 = torch.randn(N, K, generator=g, device=DEV, dtype=F64) * 0.1
    W0 = torch.randn(D, K, generator=g, device=DEV, dtype=F64) * 0.1
    return dict(row=r[nt:], col=q[nt:], val=y[nt:], trow=r[:nt], tcol=q[:nt], tval=y[:nt], X0=X0, W0=W0)


def _tau(c):
    return 1.0 / c["sigma"] ** 2


def _context(c, d, seed, **kw):
    from paper_1703_00734_gb300 import bmf
    h = {k: v.cpu().numpy() for k, v in d.items()}
    return bmf.BMF(c["N"], c["D"], h["row"], h["col"], h["val"], c["K"], _tau(c), c.get("prec", "fp32"),
                   X0=h["X0"], W0=h["W0"], test=(h["trow"], h["tcol"], h["tval"]), seed=seed, **kw)


def _factors(c, seed):
    """FP32 factors of a caller who evaluates or moves the log-joint (rows padded to 4 floats)."""
    g, K = _gen(seed, 3), c["K"]
    ld = -(-K // 4) * 4
    out = []
    for n in (c["N"], c["D"]):
        t = torch.zeros(n, ld, device=DEV)
        t[:, :K] = torch.randn(n, K, generator=g, device=DEV) * 0.7 * K ** -0.25
        out.append(t)
    return out


def _samples(c, seed):
    """Retained samples [S, R, K] of rows whose posteriors have up to `modes` separated modes (sign
    flips of a row's mean), and the clustering penalty."""
    R, S, K = c["R"], c["S"], c["K"]
    g = _gen(seed, 4)
    mean = torch.randn(R, K, generator=g, device=DEV, dtype=F64)
    flip = torch.ones(3, R, K, device=DEV, dtype=F64)
    flip[1] = -1.0
    flip[2, :, : max(1, K // 2)] = -1.0
    which = (torch.rand(S, R, generator=g, device=DEV) ** 2 * c["modes"]).long().clamp_(max=c["modes"] - 1)
    x = mean * flip[which, torch.arange(R, device=DEV)]
    return x + 0.15 * torch.randn(S, R, K, generator=g, device=DEV, dtype=F64), 0.4 * K


def _submodels(c, seed):
    """Means [J, R, K] and precisions [J, R, K, K] of J submodels of R rows: the inverse covariances
    of 6 K samples from posteriors that have seen the propagated one's data and some more."""
    R, J, K = c["R"], c["J"], c["K"]
    g = _gen(seed, 5)
    mean = torch.randn(R, K, generator=g, device=DEV, dtype=F64)
    Lam = torch.empty(J, R, K, K, device=DEV, dtype=F64)
    mu = torch.empty(J, R, K, device=DEV, dtype=F64)
    n = 6 * K
    A = torch.randn(R, K, 12, generator=g, device=DEV, dtype=F64)
    base = 4.0 * A @ A.transpose(1, 2) + torch.eye(K, device=DEV, dtype=F64)
    for j in range(J):
        B = torch.randn(R, K, 6 if j else 1, generator=g, device=DEV, dtype=F64)
        L = torch.linalg.cholesky(base + B @ B.transpose(1, 2))
        z = torch.randn(R, K, n, generator=g, device=DEV, dtype=F64)
        x = torch.linalg.solve_triangular(L.transpose(1, 2), z, upper=True)
        m = x.mean(2, keepdim=True)
        S = (x - m) @ (x - m).transpose(1, 2) / n
        P = torch.linalg.inv(S)
        Lam[j] = 0.5 * (P + P.transpose(1, 2))
        mu[j] = mean + m[:, :, 0]
    return mu, Lam


# ------------------------------------------------------------------------------------------
# prepare and run
# ------------------------------------------------------------------------------------------
def prepare(case, seed):
    c, kind = dict(case), case["kind"]
    if kind == "summaries":
        x, lam = _samples(c, seed)
        return dict(c=c, x=x, lam=lam)
    if kind == "aggregate":
        mu, Lam = _submodels(c, seed)
        return dict(c=c, mu=mu, Lam=Lam, out=torch.empty(c["R"], c["K"], device=DEV, dtype=F64))
    d = _matrix(c, seed)
    if kind == "plain":
        m = _context(c, d, seed, burnin=c["burnin"], noise=c["noise"], noise_a0=2.0,
                     noise_b0=2.0 * c["sigma"] ** 2)
        return dict(c=c, m=m, seed=seed)
    if kind == "pp":
        m = _context(c, d, seed, burnin=c["burnin"], thin=c["thin"], I=c["I"], J=c["J"])
        m.set_monitor(False)
        m.set_schedule(graph=c["graph"])
        return dict(c=c, m=m, seed=seed)
    # grad, langevin: the priors are the hyperparameters of a chain's first sweep
    m = _context(c, d, seed)
    m.sweep(0, 1)
    X, W = _factors(c, seed)
    s = dict(c=c, m=m, X=X, W=W)
    if kind == "langevin":
        s["xi"] = torch.randn(c["steps"], (c["N"] + c["D"]) * c["K"], generator=_gen(seed, 6), device=DEV)
    else:
        s["X"], s["W"] = X.requires_grad_(), W.requires_grad_()
        s["la"] = torch.tensor(math.log(_tau(c)), dtype=F64, device=DEV, requires_grad=True)
    torch.cuda.synchronize()
    return s


def _eps(c):
    return 2e-6 * c["sigma"] ** 2


def _carry(c, a):
    return a if c["prec"] == "fp64" else a.astype(np.float32)


def run(state):
    from paper_1703_00734_gb300 import bmf
    c = state["c"]
    kind = c["kind"]
    if kind == "plain":
        m = state["m"]
        m.restart(state["seed"])
        st = m.sweep(0, c["sweeps"])
        Xm, Wm, _ = m.posterior_means()
        return dict(X=_carry(c, Xm), W=_carry(c, Wm), rmse_sample=st["rmse_sample"], rmse_mean=st["rmse_mean"])
    if kind == "pp":
        m = state["m"]
        m.restart(state["seed"])
        for stage in (1, 2, 3) if c["I"] > 1 else (1, 2):
            m.stage(stage, c["sweeps"])
        rmse = m.test_rmse()
        Xm, Wm, _ = m.posterior_means()
        return dict(X=_carry(c, Xm), W=_carry(c, Wm), rmse=rmse)
    if kind == "grad":
        from paper_1703_00734_gb300.autograd import LogJoint
        X, W, la = state["X"], state["W"], state["la"]
        X.grad = W.grad = la.grad = None
        v = LogJoint.apply(state["m"], 0, X, W, la)
        v.backward()
        return dict(value=float(v), X=X.grad, W=W.grad, log_alpha=float(la.grad))
    if kind == "langevin":
        X, W = state["X"].clone(), state["W"].clone()
        _, v = state["m"].langevin(0, c["steps"], X.data_ptr(), W.data_ptr(), X.shape[1], math.log(_tau(c)),
                                   _eps(c), state["xi"].data_ptr())
        return dict(X=X, W=W, value=v)
    if kind == "summaries":
        return bmf.fit_summaries(state["x"], "gmm", state["lam"], c["C"],
                                 stream=torch.cuda.current_stream().cuda_stream)
    n = bmf.aggregate_static(c["K"], c["R"], c["J"], state["mu"].data_ptr(), state["Lam"].data_ptr(),
                             state["out"].data_ptr(), stream=torch.cuda.current_stream().cuda_stream)
    return dict(mu=state["out"], corrected=n)


# ------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------
def _row_flops(K):
    """Assembly, Cholesky and two solves of one conditional draw."""
    return 2.0 * (K * (K + 1) / 2 + K + (K ** 3 - K) / 6 + K * K)


def work(case):
    c, kind = case, case["kind"]
    if kind == "summaries":
        R, S, K, C = c["R"], c["S"], c["K"], c["C"]
        return dict(bytes=8.0 * R * (S * K + C * (1 + K + K * K) + K + K * K) + 4.0 * R * S,
                    flops=R * (3 * S * c["modes"] * 3.0 * K + 2.0 * S * K * K + (2 * c["modes"] + 1) * 2.0 * K ** 3))
    if kind == "aggregate":
        R, J, K = c["R"], c["J"], c["K"]
        return dict(bytes=8.0 * R * (J * (K * K + K) + K),
                    flops=R * ((J - 1) * (K ** 3 / 3 + 4 * K ** 3 / 3) + K ** 3 / 3 + 2.0 * (J + 1) * K * K))
    N, D, K = c["N"], c["D"], c["K"]
    M = min(c["M"], N * D // 2)
    M -= M // 10
    if kind in ("grad", "langevin"):
        n = c.get("steps", 0) + 1
        return dict(bytes=n * (2.0 * M * 8 + 8.0 * (N + D) * K * (2 if n > 1 else 1)),
                    flops=n * (2.0 * M * 4 * K + 2.0 * (N + D) * K * K))
    obs = 4 + (8 if c["prec"] == "fp64" else 4)
    gram = 2.0 * (K * (K + 1) / 2 + K)
    if kind == "plain":
        per = dict(bytes=2.0 * M * obs + 8.0 * 2 * (N + D) * K, flops=2 * M * gram + (N + D) * _row_flops(K))
    else:
        # X rows sit in J subsets and W rows in I; two of the three stages also read their
        # rows' propagated priors, and moment sums are kept after the burn-in
        I, J = c["I"], c["J"]
        rows = N * J + D * I
        keep = (c["sweeps"] - c["burnin"]) / c["thin"] / c["sweeps"]
        tri = K * (K + 1) / 2 + K
        per = dict(bytes=2.0 * M * obs + 8.0 * rows * (2 * K + 0.8 * tri + 2 * keep * tri),
                   flops=2 * M * gram + rows * (_row_flops(K) + keep * K * (K + 1)))
    return {k: v * c["sweeps"] for k, v in per.items()}


# ------------------------------------------------------------------------------------------
# the same results in 64 bits
# ------------------------------------------------------------------------------------------
_M64 = (1 << 64) - 1


def _i64(v):
    v &= _M64
    return v - (1 << 64) if v >> 63 else v


def _mulhi(a, m):
    """High 64 bits of the unsigned product of an int64 tensor (as bits) and the constant m."""
    lo = 0xFFFFFFFF
    a0, a1 = a & lo, (a >> 32) & lo
    m0, m1 = m & lo, m >> 32
    # 32 x 32 products as wrapping int64; shifts made logical by masks
    p00, p01, p10, p11 = a0 * m0, a0 * m1, a1 * m0, a1 * m1
    mid = ((p00 >> 32) & lo) + (p01 & lo) + (p10 & lo)
    return p11 + ((p01 >> 32) & lo) + ((p10 >> 32) & lo) + ((mid >> 32) & lo)


def _philox(index, t, tag, attempt, seed):
    """Philox4x64-10 (Salmon et al. 2011) with key (seed, 0) on counters (index, t, tag, attempt)."""
    x = [index, torch.full_like(index, t), torch.full_like(index, tag), torch.full_like(index, attempt)]
    m0, m1 = 0xD2E7470EE14C6C93, 0xCA5A826395121157
    k0, k1 = seed & _M64, 0
    for _ in range(10):
        h0, l0 = _mulhi(x[0], m0), x[0] * _i64(m0)
        h1, l1 = _mulhi(x[2], m1), x[2] * _i64(m1)
        x = [h1 ^ x[1] ^ _i64(k0), l1, h0 ^ x[3] ^ _i64(k1), l0]
        k0, k1 = (k0 + 0x9E3779B97F4A7C15) & _M64, (k1 + 0xBB67AE8584CAA73B) & _M64
    return x


def _unit(w, add):
    return (((w >> 11) & ((1 << 53) - 1)) + add).to(F64) * 2.0 ** -53


def _normals(n, t, tag, seed):
    w = _philox(torch.arange(-(-n // 4), device=DEV), t, tag, 0, seed)
    z = []
    for a, b in ((w[0], w[1]), (w[2], w[3])):
        r, ang = torch.sqrt(-2.0 * torch.log(_unit(a, 1))), 2.0 * math.pi * _unit(b, 0)
        z += [r * torch.cos(ang), r * torch.sin(ang)]
    return torch.stack(z, 1).reshape(-1)[:n]


def _chi2(dof, t, tag, seed):
    """2 Gamma(dof / 2) by Marsaglia & Tsang (2000), attempts on the counter's last word."""
    i = torch.arange(dof.numel(), device=DEV)
    a = 0.5 * dof
    d = torch.where(a < 1, a + 1, a) - 1.0 / 3.0
    s = 1.0 / torch.sqrt(9.0 * d)
    out, todo = torch.zeros_like(dof), torch.ones_like(dof, dtype=torch.bool)
    for j in range(64):
        w = _philox(i, t, tag, j, seed)
        x = torch.sqrt(-2.0 * torch.log(_unit(w[0], 1))) * torch.cos(2.0 * math.pi * _unit(w[1], 0))
        v = (1.0 + s * x) ** 3
        u = _unit(w[2], 1)
        ok = (v > 0) & ((u < 1 - 0.0331 * x ** 4) |
                        (torch.log(u) < 0.5 * x * x + d * (1 - v + torch.log(v.clamp(min=1e-300)))))
        g = d * v * torch.where(a < 1, _unit(w[3], 1) ** (1.0 / a), torch.ones_like(a))
        out = torch.where(todo & ok, 2.0 * g, out)
        todo &= ~ok
        if not bool(todo.any()):
            break
    return out


class _Chain:
    """One subset's Gibbs chain on reordered data, all in FP64 on the device."""

    def __init__(self, sid, r, q, y, X, W, c, seed):
        self.sid, self.X, self.W, self.c, self.seed, self.t = sid, X, W, c, seed, 0
        K = c["K"]
        self.ti = torch.tril_indices(K, K, device=DEV)
        self.prior = [None, None]
        self.S1, self.S2, self.kept = [0.0, 0.0], [0.0, 0.0], 0
        self.tau = torch.full((W.shape[0],), _tau(c), dtype=F64, device=DEV)
        self.r, self.q, self.y = r, q, y
        self.lists = []
        for a, b, n, m in ((r, q, X.shape[0], W.shape[0]), (q, r, W.shape[0], X.shape[0])):
            at = torch.argsort(a * m + b)
            ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
            ptr[1:] = torch.cumsum(torch.bincount(a, minlength=n), 0)
            self.lists.append((ptr, b[at], y[at], n, m))

    def gram(self, f, P, w):
        """sum w p p^T (full) and sum w y p of every row."""
        ptr, idx, y, n, m = self.lists[f]
        K = P.shape[1]
        one = torch.ones_like(y) if w is None else w[idx]
        prod = P[:, self.ti[0]] * P[:, self.ti[1]]
        G = torch.zeros(n, K, K, dtype=F64, device=DEV)
        b = torch.zeros(n, K, dtype=F64, device=DEV)
        if y.numel():
            A = torch.sparse_csr_tensor(ptr, idx, one, (n, m), dtype=F64)
            low = A @ prod
            G[:, self.ti[0], self.ti[1]] = low
            G[:, self.ti[1], self.ti[0]] = low
            b = torch.sparse_csr_tensor(ptr, idx, one * y, (n, m), dtype=F64) @ P
        return G, b

    def hyper(self, f):
        """Normal-Wishart posterior (centred scatter) and its Bartlett draw."""
        A = self.X if f == 0 else self.W
        n, K = A.shape
        tag = self.sid * 256 + f * 16
        z = _normals(K * (K - 1) // 2 + K, self.t, tag + 2, self.seed)
        chi = _chi2(K + n - torch.arange(K, device=DEV, dtype=F64), self.t, tag + 1, self.seed)
        eye = torch.eye(K, dtype=F64, device=DEV)
        xbar = A.mean(0)
        Ac = A - xbar
        Winv = eye + Ac.T @ Ac + 2.0 * n / (2.0 + n) * torch.outer(xbar, xbar)
        L = torch.linalg.cholesky(torch.linalg.inv(Winv))
        B = torch.diag(torch.sqrt(chi))
        low = torch.tril_indices(K, K, -1, device=DEV)
        B[low[0], low[1]] = z[: K * (K - 1) // 2]
        LA = L @ B
        Lam = LA @ LA.T
        mu = n * xbar / (2.0 + n) + torch.linalg.solve_triangular(
            math.sqrt(2.0 + n) * LA.T, z[K * (K - 1) // 2:, None], upper=True)[:, 0]
        return mu, Lam

    def half(self, f, hyp):
        A, P = (self.X, self.W) if f == 0 else (self.W, self.X)
        n, K = A.shape
        noisy = self.c.get("noise", "fixed") != "fixed"
        G, b = self.gram(f, P, self.tau if (f == 0 and noisy) else None)
        if not (f == 0 and noisy):
            t = self.tau if f == 1 else self.tau[:1]
            G, b = G * t[:, None, None], b * t[:, None]
        if self.prior[f] is not None:
            mu, L0 = self.prior[f]
            G, b = G + L0, b + (L0 @ mu[:, :, None])[:, :, 0]
        else:
            mu, L0 = hyp
            G, b = G + L0, b + L0 @ mu
        L = torch.linalg.cholesky(G)
        z = _normals(n * K, self.t, self.sid * 256 + f * 16 + 3, self.seed).reshape(n, K, 1)
        v = torch.linalg.solve_triangular(L, b[:, :, None], upper=False)
        new = torch.linalg.solve_triangular(L.transpose(1, 2), v + z, upper=True)[:, :, 0]
        if f == 0:
            self.X = new
        else:
            self.W = new

    def sweep(self):
        c = self.c
        self.t += 1
        hyp = [None if self.prior[f] is not None else self.hyper(f) for f in (0, 1)]
        self.half(0, hyp[0])
        self.half(1, hyp[1])
        if c.get("noise", "fixed") == "column":
            d = self.W.shape[0]
            e2 = torch.zeros(d, dtype=F64, device=DEV)
            e = self.y - (self.X[self.r] * self.W[self.q]).sum(1)
            e2.index_add_(0, self.q, e * e)
            n = torch.bincount(self.q, minlength=d).to(F64)
            self.tau = _chi2(4.0 + n, self.t, self.sid * 256 + 20, self.seed) / (4.0 * c["sigma"] ** 2 + e2)
        if self.t > c["burnin"] and (self.t - c["burnin"] - 1) % c.get("thin", 1) == 0:
            self.kept += 1
            for f, A in enumerate((self.X, self.W)):
                self.S1[f] = self.S1[f] + A
                if c["kind"] == "pp":
                    self.S2[f] = self.S2[f] + A[:, :, None] * A[:, None, :]

    def matched(self, f):
        m = self.S1[f] / self.kept
        L = torch.linalg.inv(self.S2[f] / self.kept - m[:, :, None] * m[:, None, :])
        return m, 0.5 * (L + L.transpose(1, 2))


def _combine(mu, Lam):
    """Eq. 14 with the eigenvalue correction of Algorithm 2; submodel 0 was propagated."""
    J, K = mu.shape[0], mu.shape[2]
    L1 = Lam[0]
    eps = 1e-6 * torch.clamp(torch.diagonal(L1, dim1=1, dim2=2).mean(1), min=1.0)
    tot = (2.0 - J) * L1
    rhs = (tot @ mu[0][:, :, None])[:, :, 0]
    n = 0
    for j in range(1, J):
        dif = Lam[j] - L1
        bad = torch.linalg.cholesky_ex(dif)[1] != 0
        low = torch.zeros(dif.shape[0], dtype=F64, device=DEV)
        if bool(bad.any()):
            low[bad] = torch.linalg.eigvalsh(dif[bad])[:, 0].abs() + eps[bad]
        n += int(bad.sum())
        Lj = Lam[j] + low[:, None, None] * torch.eye(K, dtype=F64, device=DEV)
        tot = tot + Lj
        rhs = rhs + (Lj @ mu[j][:, :, None])[:, :, 0]
    return torch.linalg.solve(tot, rhs[:, :, None])[:, :, 0], n


def _order(idx, n):
    return torch.argsort(-torch.bincount(idx, minlength=n), stable=True)


def _exact_chain(c, seed):
    d = _matrix(c, seed)
    N, D, I, J = c["N"], c["D"], c.get("I", 1), c.get("J", 1)
    row, col = d["row"].long(), d["col"].long()
    off = d["val"].mean()
    rp, cp = _order(row, N), _order(col, D)
    rr, cr = torch.empty_like(rp), torch.empty_like(cp)
    rr[rp], cr[cp] = torch.arange(N, device=DEV), torch.arange(D, device=DEV)
    r, q, y = rr[row], cr[col], d["val"] - off
    X0, W0 = d["X0"][rp], d["W0"][cp]
    rb, cb = [k * N // I for k in range(I + 1)], [k * D // J for k in range(J + 1)]

    def chain(i, j):
        at = (r >= rb[i]) & (r < rb[i + 1]) & (q >= cb[j]) & (q < cb[j + 1])
        return _Chain(i * J + j, r[at] - rb[i], q[at] - cb[j], y[at], X0[rb[i]:rb[i + 1]], W0[cb[j]:cb[j + 1]],
                      c, seed)

    def back(Xm, Wm):
        Xo, Wo = torch.empty_like(Xm), torch.empty_like(Wm)
        Xo[rp], Wo[cp] = Xm, Wm
        return Xo, Wo

    return d, off, chain, back


def _rmse(d, off, X, W):
    s = 0.0
    for a in range(0, d["trow"].numel(), 1 << 21):
        e = slice(a, a + (1 << 21))
        p = off + (X[d["trow"][e].long()] * W[d["tcol"][e].long()]).sum(1)
        s += float(((d["tval"][e] - p) ** 2).sum())
    return math.sqrt(s / max(1, d["trow"].numel()))


def _exact_plain(c, seed):
    d, off, chain, back = _exact_chain(c, seed)
    ch = chain(0, 0)
    tr, tc = d["trow"].long(), d["tcol"].long()
    ysum = torch.zeros(tr.numel(), dtype=F64, device=DEV)
    sample = 0.0
    for t in range(c["sweeps"]):
        kept = ch.kept
        ch.sweep()
        if ch.kept > kept or t + 1 == c["sweeps"]:
            X, W = back(ch.X, ch.W)
            p = torch.cat([(X[tr[a:a + (1 << 21)]] * W[tc[a:a + (1 << 21)]]).sum(1)
                           for a in range(0, tr.numel(), 1 << 21)])
            sample = float(((d["tval"] - off - p) ** 2).mean().sqrt())
            if ch.kept > kept:
                ysum += p
    mean = float(((d["tval"] - off - ysum / ch.kept) ** 2).mean().sqrt())
    X, W = back(ch.S1[0] / ch.kept, ch.S1[1] / ch.kept)
    return dict(X=X, W=W, rmse_sample=sample, rmse_mean=mean)


def _exact_pp(c, seed):
    d, off, chain, back = _exact_chain(c, seed)
    I, J = c["I"], c["J"]
    done = {}
    stages = [[(0, 0)], [(i, 0) for i in range(1, I)] + [(0, j) for j in range(1, J)],
              [(i, j) for i in range(1, I) for j in range(1, J)]]
    for k, stage in enumerate(stages):
        for i, j in stage:
            ch = chain(i, j)
            if j > 0 and k:      # X^(i) from (i, 0)
                ch.prior[0] = done[i, 0][0]
                ch.X = ch.prior[0][0].clone()
            if i > 0 and k:      # W^(j) from (0, j)
                ch.prior[1] = done[0, j][1]
                ch.W = ch.prior[1][0].clone()
            for _ in range(c["sweeps"]):
                ch.sweep()
            done[i, j] = (ch.matched(0), ch.matched(1), ch.S1[0] / ch.kept, ch.S1[1] / ch.kept)
    X, W = [], []
    for i in range(I):
        X.append(done[i, 0][2] if J == 1 else _combine(*(torch.stack([done[i, j][0][p] for j in range(J)])
                                                         for p in (0, 1)))[0])
    for j in range(J):
        W.append(done[0, j][3] if I == 1 else _combine(*(torch.stack([done[i, j][1][p] for i in range(I)])
                                                         for p in (0, 1)))[0])
    X, W = back(torch.cat(X), torch.cat(W))
    return dict(X=X, W=W, rmse=_rmse(d, off, X, W))


def _exact_logjoint(c, seed):
    """A function of (X, W) in local order: value, gradients and d value / d log alpha."""
    d, off, chain, _ = _exact_chain(dict(c, burnin=0), seed)
    ch = chain(0, 0)
    ch.t = 1
    (mx, Lx), (mw, Lw) = ch.hyper(0), ch.hyper(1)
    a, n = _tau(c), ch.y.numel()

    def at(X, W):
        r2 = 0.0
        gX, gW = -(X @ Lx - Lx @ mx), -(W @ Lw - Lw @ mw)
        quad = float((X * (X @ Lx)).sum() - 2 * (X @ (Lx @ mx)).sum() + (W * (W @ Lw)).sum()
                     - 2 * (W @ (Lw @ mw)).sum())
        for b in range(0, n, 1 << 20):
            r, q = ch.r[b:b + (1 << 20)], ch.q[b:b + (1 << 20)]
            x, w = X[r], W[q]
            e = ch.y[b:b + (1 << 20)] - (x * w).sum(1)
            r2 += float((e * e).sum())
            gX.index_add_(0, r, a * e[:, None] * w)
            gW.index_add_(0, q, a * e[:, None] * x)
        return -0.5 * a * r2 + 0.5 * n * math.log(a) - 0.5 * quad, gX, gW, 0.5 * n - 0.5 * a * r2

    return at


def _exact_grad(c, seed):
    X, W = (t[:, :c["K"]].to(F64) for t in _factors(c, seed))
    v, gX, gW, ga = _exact_logjoint(c, seed)(X, W)
    pad = -(-c["K"] // 4) * 4 - c["K"]
    return dict(value=v, X=torch.nn.functional.pad(gX, (0, pad)), W=torch.nn.functional.pad(gW, (0, pad)),
                log_alpha=ga)


def _exact_langevin(c, seed):
    N, D, K = c["N"], c["D"], c["K"]
    X, W = (t[:, :K].to(F64) for t in _factors(c, seed))
    xi = torch.randn(c["steps"], (N + D) * K, generator=_gen(seed, 6), device=DEV).to(F64)
    at = _exact_logjoint(c, seed)
    eps = _eps(c)
    v, gX, gW, _ = at(X, W)
    for k in range(c["steps"]):
        X = X + 0.5 * eps * gX + math.sqrt(eps) * xi[k, : N * K].reshape(N, K)
        W = W + 0.5 * eps * gW + math.sqrt(eps) * xi[k, N * K:].reshape(D, K)
        v, gX, gW, _ = at(X, W)
    pad = -(-K // 4) * 4 - K
    return dict(X=torch.nn.functional.pad(X, (0, pad)), W=torch.nn.functional.pad(W, (0, pad)), value=v)


def _exact_summaries(c, seed):
    x, lam = _samples(c, seed)
    S, R, K = x.shape
    C, most = c["C"], 24
    x = x.transpose(0, 1).contiguous()
    rows = torch.arange(R, device=DEV)
    cen = torch.full((R, most, K), math.inf, dtype=F64, device=DEV)
    cen[:, 0] = x[:, 0]
    n = torch.ones(R, dtype=torch.int64, device=DEV)
    prev = torch.full((R, S), -1, device=DEV)
    live = torch.ones(R, dtype=torch.bool, device=DEV)
    slot = torch.arange(most, device=DEV)
    for _ in range(100):
        now = torch.empty_like(prev)
        for i in range(S):
            dist = ((x[:, i:i + 1] - cen) ** 2).sum(2)
            dist = torch.where(slot[None] < n[:, None], dist, torch.full_like(dist, math.inf))
            best, which = dist.min(1)
            new = (best > lam) & live
            if bool(new.any()):
                if int(n.max()) >= most:
                    return None
                cen[rows[new], n[new]] = x[new, i]
                which = torch.where(new, n, which)
                n = n + new
            now[:, i] = which
        cnt = torch.zeros(R, most, dtype=torch.int64, device=DEV).scatter_add_(1, now, torch.ones_like(now))
        to = torch.cumsum((cnt > 0).long(), 1) - 1
        now = to.gather(1, now)
        cnt = torch.zeros(R, most, dtype=torch.int64, device=DEV).scatter_add_(1, now, torch.ones_like(now))
        tot = torch.zeros(R, most, K, dtype=F64, device=DEV).scatter_add_(1, now[:, :, None].expand(R, S, K), x)
        ncen = torch.where(cnt[:, :, None] > 0, tot / cnt[:, :, None], torch.full_like(tot, math.inf))
        same = (now == prev).all(1)
        up = live
        cen[up], n = ncen[up], torch.where(up, (cnt > 0).sum(1), n)
        prev = torch.where(up[:, None], now, prev)
        live = live & ~same
        if not bool(live.any()):
            break
    size = torch.zeros(R, most, dtype=torch.int64, device=DEV).scatter_add_(1, prev, torch.ones_like(prev))
    pi = torch.zeros(R, C, dtype=F64, device=DEV)
    mu = torch.zeros(R, C, K, dtype=F64, device=DEV)
    Lam = torch.zeros(R, C, K, K, dtype=F64, device=DEV)
    cov = torch.zeros(R, C, K, K, dtype=F64, device=DEV)
    got = torch.zeros(R, dtype=torch.int64, device=DEV)

    def gauss(w):
        k = w.sum(1)
        m = (w[:, :, None] * x).sum(1) / k[:, None]
        e = (x - m[:, None]) * w[:, :, None]
        return k, m, e.transpose(1, 2) @ e / k[:, None, None]

    left = size.clone()
    for k in range(C):
        big, which = left.max(1)
        left = left.scatter(1, which[:, None], -1)
        use = big >= K + 1
        if not bool(use.any()):
            continue
        sz, m, S2 = gauss((prev == which[:, None]).to(F64))
        r = rows[use]
        pi[r, got[use]], mu[r, got[use]], cov[r, got[use]] = sz[use], m[use], S2[use]
        Lam[r, got[use]] = torch.linalg.inv(S2[use])
        got = got + use
    none = got == 0
    if bool(none.any()):
        _, m, S2 = gauss(torch.ones(R, S, dtype=F64, device=DEV))
        pi[none, 0], mu[none, 0], cov[none, 0] = 1.0, m[none], S2[none]
        Lam[none, 0] = torch.linalg.inv(S2[none])
    pi = pi / pi.sum(1, keepdim=True)
    pm = (pi[:, :, None] * mu).sum(1)
    e = mu - pm[:, None]
    P = (pi[:, :, None, None] * (cov + e[:, :, :, None] * e[:, :, None, :])).sum(1)
    return dict(pi=pi, mu=mu, Lam=Lam, pooled_mu=pm, pooled_Lam=torch.linalg.inv(P), assign=prev.to(torch.int32))


def exact(case, seed):
    c, kind = dict(case), case["kind"]
    if kind == "pp":
        # about 20 seconds where the run has more than this many row draws and entries
        cost = c["sweeps"] * (c["N"] * c["J"] + c["D"] * c["I"] + 0.1 * c["M"]) * c["K"]
        return None if cost > 4e8 or c["I"] * c["J"] * c["sweeps"] > 4000 else _exact_pp(c, seed)
    if kind == "plain":
        return _exact_plain(c, seed)
    if kind == "grad":
        return _exact_grad(c, seed)
    if kind == "langevin":
        return _exact_langevin(c, seed)
    if kind == "summaries":
        return _exact_summaries(c, seed)
    mu, Lam = _submodels(c, seed)
    out, n = _combine(mu, Lam)
    return dict(mu=out, corrected=n)
