"""Performance cases of the CRBM-aided Monte Carlo library.

Each case is work a user's program does through the public layer
(`paper_2008_05401_gb300`): load filters, create jobs, upload lattices, run
proposals, tempering cycles or local sweeps, read lattices and observables
back, train filters, estimate autocorrelation times.  Sizes are those of the
repository's workloads, benchmark and tests.  `exact` restates the method in
plain torch / numpy FP64 (its own Philox, convolutions, spectra, exchanges,
ADAM) and returns what `run` returns.
"""
from __future__ import annotations

import math
import os
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

import paper_2008_05401_gb300 as crbm
from paper_2008_05401_gb300 import FP64, ISING, KITAEV, MIXED, trainer

DEV = "cuda:0"
EDGE = 3                # unshared kernels per side of the open-boundary model's CRBM
BATCH, LR, B1, B2, EPS = 20, 1e-3, 0.9, 0.999, 1e-8   # the trainer's defaults
PACKAGE = os.path.dirname(os.path.abspath(crbm.__file__))


def listed():
    return [
        # the small Ising workload: 16 chains of 8 x 8 in plain FP64, a first look at a new set of filters
        dict(name="ising_small_fp64", kind="ising", Ls="8", chains=16, K=2, k=3, S=100, prec="fp64"),
        # the batch Ising workload end to end: upload of every lattice, one batched run, read-back
        dict(name="ising_batch", kind="ising", Ls="128,64,32,16", chains=4096, K=4, k=5, S=10, prec="mixed"),
        # sides of the paper's timing table that are no power of two, its 2 filters of 5 x 5
        dict(name="ising_L24", kind="ising", Ls="24", chains=1024, K=2, k=5, S=20, prec="mixed"),
        # a served request at the largest side: few chains, many sequential proposals
        dict(name="ising_L256_serving", kind="ising", Ls="256", chains=16, K=4, k=5, S=40, prec="mixed"),
        # the small Kitaev workload (72 sites), mixed precision
        dict(name="kitaev_L6", kind="kitaev", Ls="6", chains=1024, K=4, k=3, S=8, prec="mixed"),
        # the same in plain FP64, the precision of its definition
        dict(name="kitaev_L6_fp64", kind="kitaev", Ls="6", chains=1024, K=4, k=3, S=4, prec="fp64"),
        # the batch Kitaev workload: three sides in one call, mixed precision
        dict(name="kitaev_batch", kind="kitaev", Ls="12,10,8", chains=683, K=4, k=3, S=3, prec="mixed"),
        # the paper's Kitaev protocol: tempering with 4 Gibbs steps per correction
        dict(name="kitaev_tempering", kind="tempering", model="kitaev", L=8, chains=1024, K=4, k=3, g=4, S=6,
             prec="mixed"),
        # open boundaries with three unshared kernels per side (FP64 is its only precision)
        dict(name="kitaev_open", kind="open", L=8, chains=1024, K=2, k=5, S=4),
        # the paper's baseline sampler: checkerboard Metropolis sweeps with an energy trace
        dict(name="ising_sweeps", kind="sweeps", L=64, chains=512, S=100, exchange=False),
        # autocorrelation times of one energy trace of 1024 chains
        dict(name="autocorr", kind="autocorr", series=1024, length=2000, tau=28.0),
        # one training epoch of 24 temperatures side by side
        dict(name="train_epoch", kind="train", problems=24, L=8, K=2, k=5, samples=10000),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    what = rng.choice(["ising", "ising", "ising", "kitaev", "kitaev", "kitaev", "tempering", "open", "sweeps",
                       "autocorr", "train"])
    if what == "ising":
        prec = rng.choice(["mixed", "mixed", "fp64"])
        L = rng.choice([8, 12, 16, 20, 24, 30, 31, 32, 64, 96, 128, 256])
        K, k = rng.choice([(2, 3), (4, 3), (2, 5), (4, 5)])
        # FP64 proposals cost about 60 times as much: fewer sites for the same pass
        sites = 4e7 if prec == "mixed" else 1e6
        n = _log(rng, 1, max(1, min(4096, int(sites / (L * L)))))
        return dict(kind="ising", Ls=str(L), chains=n, K=K, k=k, S=_log(rng, 1, 60), prec=prec)
    if what == "kitaev":
        K, k = rng.choice([(4, 3), (2, 3), (4, 3)])
        L = rng.choice([4, 5, 6, 7, 8, 9, 10, 11, 12])
        return dict(kind="kitaev", Ls=str(L), chains=_log(rng, 8, 1500 if L > 8 else 2048), K=K, k=k,
                    S=rng.randint(1, 3), prec=rng.choice(["mixed", "mixed", "fp64"]))
    if what == "tempering":
        if rng.random() < 0.4:
            return dict(kind="tempering", model="ising", L=rng.choice([8, 16, 24, 32]), chains=_log(rng, 31, 4096),
                        K=4, k=5, g=rng.randint(1, 4), S=rng.randint(2, 12), prec=rng.choice(["mixed", "fp64"]))
        return dict(kind="tempering", model="kitaev", L=rng.choice([4, 6, 8]), chains=_log(rng, 24, 1024), K=4, k=3,
                    g=rng.randint(1, 6), S=rng.randint(2, 6), prec=rng.choice(["mixed", "fp64"]))
    if what == "open":
        return dict(kind="open", L=rng.choice([6, 7, 8, 10]), chains=_log(rng, 8, 1024), K=2, k=rng.choice([3, 5]),
                    S=rng.randint(1, 3))
    if what == "sweeps":
        return dict(kind="sweeps", L=rng.choice([8, 16, 30, 32, 64, 128]), chains=_log(rng, 16, 1024),
                    S=_log(rng, 10, 120), exchange=rng.random() < 0.4)
    if what == "autocorr":
        return dict(kind="autocorr", series=_log(rng, 3, 1100), length=_log(rng, 200, 4000),
                    tau=round(math.exp(rng.uniform(math.log(1.5), math.log(30.0))), 2))
    return dict(kind="train", problems=_log(rng, 1, 30), L=rng.choice([4, 6, 8, 10, 12]), K=rng.choice([1, 2, 4]),
                k=rng.choice([3, 5] if rng.random() < 0.8 else [2, 4]), samples=_log(rng, 500, 4000))


# ---------------------------------------------------------------- inputs
def _sides(case):
    return [int(x) for x in case["Ls"].split(",")]


def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1009 + salt)
    return g


def _filters(case, seed):
    """The batch Ising workload's trained filters where the shape is theirs, else Gaussian ones of the workloads' widths."""
    K, k = case["K"], case["k"]
    ising = case["kind"] == "ising" or case.get("model") == "ising"
    if ising and (K, k) == (4, 5):
        d = np.load(os.path.join(PACKAGE, "data", "ising_cd1_L16_K4_k5.npz"))
        return d["W"], float(d["vb"]), d["hb"]
    g = np.random.default_rng([int(seed), 7])
    std = 0.1 if ising else 0.05
    lead = (2 * EDGE + 1, K, k, k) if case["kind"] == "open" else (K, k, k)
    return g.normal(0.0, std, lead), float(g.normal(0.0, std)), g.normal(0.0, std, K)


def _ladder(case, n):
    if case["kind"] in ("kitaev", "open") or case.get("model") == "kitaev":
        Ts = 0.005 * 200.0 ** (np.arange(24) / 23.0)
    else:
        Ts = 1.5 + 2.0 * np.arange(32) / 31.0
    return Ts[np.arange(n) % len(Ts)]


def _ising_lattices(n, L, T, seed, salt):
    """(n, L, L) uint8 lattices with the domains of their temperature: 30 checkerboard heat-bath sweeps from random ones."""
    g = _gen(seed, salt)
    s = torch.randint(0, 2, (n, L, L), generator=g, device=DEV, dtype=torch.int8).float().mul_(2).sub_(1)
    beta = torch.as_tensor(1.0 / T, device=DEV, dtype=torch.float32)[:, None, None]
    i = torch.arange(L, device=DEV)
    black = ((i[:, None] + i[None, :]) % 2 == 0)[None]
    for sweep in range(60):
        nn = s.roll(1, 1) + s.roll(-1, 1) + s.roll(1, 2) + s.roll(-1, 2)
        up = torch.rand(s.shape, generator=g, device=DEV) < torch.sigmoid(2.0 * beta * nn)
        s = torch.where(black if sweep % 2 == 0 else ~black, up.float().mul_(2).sub_(1), s)
    return (s > 0).to(torch.uint8)


def _lattices(case, n, L, T, seed, salt):
    if case["kind"] in ("kitaev", "open") or case.get("model") == "kitaev":
        return torch.randint(0, 2, (n, L, L), generator=_gen(seed, salt), device=DEV, dtype=torch.uint8)
    return _ising_lattices(n, L, T, seed, salt)


def _pack(v):
    """(n, L, L) 0/1 tensor -> (n, ceil(L*L/32)) uint32 array, site n at bit n % 32 of word n // 32."""
    n, N = v.shape[0], v.shape[1] * v.shape[2]
    Wd = (N + 31) // 32
    flat = torch.zeros((n, Wd * 32), dtype=torch.int64, device=v.device)
    flat[:, :N] = v.reshape(n, N)
    words = (flat.view(n, Wd, 32) << torch.arange(32, device=v.device)).sum(2)
    return words.cpu().numpy().astype(np.uint32)


def _pinned(a, dtype):
    """The array in pinned host memory, as a program that uploads and reads back in a loop keeps it."""
    t = torch.empty(a if isinstance(a, tuple) else a.shape, dtype=dtype, pin_memory=True).numpy()
    t = t.view(np.uint32) if dtype == torch.int32 else t
    if not isinstance(a, tuple):
        t[...] = a
    return t


def _series(case, seed):
    """(length, series) AR(1) traces with integrated autocorrelation time case["tau"]."""
    rho = (2.0 * case["tau"] - 1.0) / (2.0 * case["tau"] + 1.0)
    g = _gen(seed, 3)
    eta = torch.randn((case["length"], case["series"]), generator=g, device=DEV, dtype=torch.float64)
    x = torch.empty_like(eta)
    x[0] = eta[0]
    for t in range(1, case["length"]):
        torch.add(eta[t], x[t - 1], alpha=rho, out=x[t])
    return x * (4096.0 * 0.1) - 4096.0 * 1.4       # the scale of an energy trace at L = 64


def _training_set(case, seed):
    """Per problem: lattices, targets beta E at its temperature, visiting order, initial parameters."""
    P, L, n, K, k = (case[x] for x in ("problems", "L", "samples", "K", "k"))
    g = _gen(seed, 5)
    T = 1.5 + 0.05 * np.arange(P)
    vs, ts, orders, thetas = [], [], [], []
    for i in range(P):
        v = torch.randint(0, 2, (n, L, L), generator=g, device=DEV, dtype=torch.uint8)
        s = 2.0 * v.double() - 1.0
        E = -(s * (s.roll(-1, 1) + s.roll(-1, 2))).sum((1, 2))
        vs.append(v)
        ts.append(E / T[i])
        orders.append(torch.randperm(n, generator=g, device=DEV).to(torch.int32))
        th = torch.zeros(K * k * k + 1 + K, dtype=torch.float64, device=DEV)
        th[:K * k * k] = torch.randn(K * k * k, generator=g, device=DEV, dtype=torch.float64) * (2.0 / (K * k * k))
        thetas.append(th)
    return vs, ts, orders, thetas


# ------------------------------------------------------------- preparation
class State:
    """What a program keeps: a context, its jobs and buffers, and the pass over them."""

    def __init__(self, ctx, go, **kept):
        self.ctx, self.go, self.kept = ctx, go, kept

    def __del__(self):
        self.ctx.close()


def _result(job, energies=False):
    bits, _ = job.state()
    sums, acc, _ = job.observables()
    out = {"bits": bits.view(np.int32), "sums": sums, "accepts": acc}
    if energies:
        out["logpi"], out["F"], out["E"] = job.energies()
    return out


def prepare(case, seed):
    kind = case["kind"]
    ctx = crbm.Context(0)
    if kind == "autocorr":
        x = _series(case, seed)
        return State(ctx, lambda: list(ctx.autocorr(x)), x=x)
    if kind == "train":
        vs, ts, orders, thetas = _training_set(case, seed)
        xs = [torch.from_numpy(_pack(v).view(np.int32)).to(DEV) for v in vs]
        probs = []
        for th in thetas:
            probs.append(trainer.Problem.new(ctx, case["K"], case["k"], case["L"], th.cpu().numpy()))

        def go():
            losses = trainer.train_epochs(ctx, probs, xs, ts, orders, BATCH, LR, B1, B2, EPS)
            return {"theta": torch.stack([p.theta for p in probs]), "m": torch.stack([p.m for p in probs]),
                    "v": torch.stack([p.v for p in probs]), "t": torch.stack([p.t for p in probs]),
                    "losses": torch.stack(losses)}
        return State(ctx, go, xs=xs, ts=ts, orders=orders, probs=probs)
    if kind == "sweeps":
        n, L = case["chains"], case["L"]
        T = _ladder(case, n)
        mid = ctx.load_model(ISING, np.zeros((1, 2, 2)), 0.0, np.zeros(1))
        job = ctx.new_job(mid, ISING, L, T, (1.0,), int(seed), 0, _pack(_ising_lattices(n, L, T, seed, 1)), FP64)

        def go():
            trace = job.set_trace(case["S"])
            job.local_run(case["S"], exchange=case["exchange"])
            return {**_result(job), "trace": trace}
        return State(ctx, go)
    W, vb, hb = _filters(case, seed)
    prec = FP64 if case.get("prec", "fp64") == "fp64" else MIXED
    if kind == "open":
        n, L = case["chains"], case["L"]
        T = _ladder(case, n)
        mid = ctx.load_lcrbm(KITAEV, W, vb, hb)
        job = ctx.new_job(mid, KITAEV, L, T, (1.0, 1.0, 1.0), int(seed), 0, _pack(_lattices(case, n, L, T, seed, 1)))

        def go():
            job.run(case["S"])
            return _result(job, energies=True)
        return State(ctx, go)
    if kind == "tempering":
        n, L = case["chains"], case["L"]
        model, J = (ISING, (1.0,)) if case["model"] == "ising" else (KITAEV, (1.0, 1.0, 1.0))
        T = _ladder(case, n)
        mid = ctx.load_model(model, W, vb, hb)
        phys, rbm = (ctx.new_job(mid, model, L, T, J, int(seed) + i, i * n, _pack(_lattices(case, n, L, T, seed, 1 + i)),
                                 prec) for i in (0, 1))

        def go():
            ctx.pt_run(phys, rbm, case["S"], g=case["g"], precision=prec)
            return {"phys": _result(phys, energies=True), "rbm": rbm.state()[0].view(np.int32)}
        return State(ctx, go)
    model, J = (ISING, (1.0,)) if kind == "ising" else (KITAEV, (1.0, 1.0, 1.0))
    n = case["chains"]
    T = _ladder(case, n)
    mid = ctx.load_model(model, W, vb, hb)
    sides = _sides(case)
    first = [_pack(_lattices(case, n, L, T, seed, 1 + i)) for i, L in enumerate(sides)]
    jobs = [ctx.new_job(mid, model, L, T, J, int(seed), i * n, b, prec) for i, (L, b) in enumerate(zip(sides, first))]
    if len(jobs) == 1:
        def go():
            jobs[0].run(case["S"], precision=prec)
            return _result(jobs[0], energies=prec == FP64)
        return State(ctx, go)
    if model == KITAEV:
        def go():
            ctx.run_batch(jobs, case["S"], precision=prec)
            return [_result(j) for j in jobs]
        return State(ctx, go)
    # the request loop of the batch workload: lattices come from pinned host memory and go back there
    up = [_pinned(b, torch.int32) for b in first]
    down = [_pinned(b.shape, torch.int32) for b in first]
    sums = [_pinned((n, crbm.binding.NOBS), torch.float64) for _ in jobs]

    def go():
        ctx.write_states(jobs, up, [0] * len(jobs), prec)
        ctx.run_batch(jobs, case["S"], precision=prec)
        ctx.read_states(jobs, down, sums)
        return {"bits": [b.view(np.int32) for b in down], "sums": sums}
    return State(ctx, go)


def run(state):
    return state.go()


# -------------------------------------------------------------------- work
def work(case):
    """Bytes: every input read and every output written once.  Flops: two per multiply-add of the method's
    convolutions (hidden and visible pass of each Gibbs step, the pre-activations of F), (8/3) N^3 per Kitaev
    spectrum, one multiply-add per lag and step of an autocorrelation."""
    kind = case["kind"]
    if kind == "autocorr":
        n, t = case["series"], case["length"]
        return {"bytes": 8.0 * n * t + 16.0 * n, "flops": 2.0 * n * t * min(t - 1.0, 5.0 * case["tau"])}
    if kind == "train":
        N, P = case["L"] ** 2, case["problems"]
        params = case["K"] * case["k"] ** 2 + 1 + case["K"]
        return {"bytes": P * (case["samples"] * (4.0 * ((N + 31) // 32) + 12.0) + 48.0 * params),
                "flops": 4.0 * P * case["samples"] * N * case["K"] * case["k"] ** 2}
    n, S = case["chains"], case["S"]
    total = {"bytes": 0.0, "flops": 0.0}
    for L in _sides(case) if "Ls" in case else [case["L"]]:
        N = L * L
        state = 4.0 * ((N + 31) // 32) + 8.0 * (1 + 4 + 3 + 1)     # lattice; T, sums, energies, accepts
        total["bytes"] += 2.0 * n * state * (2 if kind == "tempering" else 1)
        if kind == "sweeps":
            total["bytes"] += 8.0 * n * S
            total["flops"] += 10.0 * n * N * S                     # neighbour sum, comparison, energy per site
            continue
        total["flops"] += 2.0 * n * S * N * case["K"] * case["k"] ** 2 * (2 * case.get("g", 1) + 1)
        if kind in ("kitaev", "open") or case.get("model") == "kitaev":
            total["flops"] += n * S * 8.0 / 3.0 * N ** 3
    return total


# ------------------------------------------------- the method in plain FP64
M32 = 0xFFFFFFFF
TAG_ACCEPT, TAG_SWAP, TAG_TEMP, TAG_LOCAL = 0xFFFFFFFE, 0xFFFFFFFD, 0xFFFFFFFC, 0xFFFFFFFB


def _philox(q, tag, step, cid, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors holding 32-bit words: counter (q, tag, step, cid)."""
    q, cid = torch.broadcast_tensors(q, cid)
    c = [q, torch.full_like(q, tag), torch.full_like(q, step), cid]
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]              # the low 64 bits, wrapped
        c = [((p1 >> 32) & M32) ^ c[1] ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c[3] ^ k1, p0 & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _uniform_plane(L, tag, step, cid, seed):
    N = L * L
    q = torch.arange((N + 3) // 4, device=DEV)
    w = torch.stack(_philox(q[None], tag, step, cid[:, None], seed), 2).reshape(len(cid), -1)[:, :N]
    return ((w.double() + 0.5) * 2.0 ** -32).view(len(cid), L, L)


def _log_uniform(tag, step, cid, seed):
    return torch.log((_philox(torch.zeros_like(cid), tag, step, cid, seed)[0].double() + 0.5) * 2.0 ** -32)


class Chains:
    """n chains of one job: lattices and their F, log pi, E, observables."""

    def __init__(self, model, W, vb, hb, v, T, seed, cid0):
        self.kitaev, self.open = model == KITAEV, W.ndim == 4
        self.vb, self.hb, self.seed = vb, hb, seed
        self.K, self.k, self.L = W.shape[-3], W.shape[-1], v.shape[-1]
        self.v = v.double()
        self.cid = cid0 + torch.arange(len(v), device=DEV)
        self.beta = torch.as_tensor(1.0 / T, device=DEV)
        self.W = {}                               # taps: a number, or one value per column (open columns)
        j = np.arange(self.L)
        cls = np.where(j < EDGE, j, np.where(j >= self.L - EDGE, 2 * EDGE + j - self.L, 2 * EDGE))
        for f in range(self.K):
            for a in range(self.k):
                for b in range(self.k):
                    self.W[f, a, b] = (torch.as_tensor(np.where(j + b < self.L, W[cls, f, a, b], 0.0), device=DEV)
                                       if self.open else float(W[f, a, b]))
        self.sums = torch.zeros((len(v), 4), dtype=torch.float64, device=DEV)
        self.acc = torch.zeros(len(v), dtype=torch.int64, device=DEV)
        self.step = 0
        self.now = self.evaluate(self.v)

    def pre(self, v, f):
        x = torch.full_like(v, float(self.hb[f]))
        for a in range(self.k):
            for b in range(self.k):
                x += self.W[f, a, b] * v.roll((-a, -b), (1, 2))
        return x

    def gibbs(self, g):
        v, t = self.v, self.step
        for s in range(g):
            x = torch.full_like(v, self.vb)
            for f in range(self.K):
                h = (_uniform_plane(self.L, s * (self.K + 1) + f, t, self.cid, self.seed)
                     < torch.sigmoid(self.pre(v, f))).double()
                for a in range(self.k):
                    for b in range(self.k):
                        x += (self.W[f, a, b] * h).roll((a, b), (1, 2))
            v = (_uniform_plane(self.L, s * (self.K + 1) + self.K, t, self.cid, self.seed) < torch.sigmoid(x)).double()
        return v

    def spectrum(self, v):
        """Singular values of M_bw = 2 J u_bw: z-bond (i, j), x-bond to (i + 1, j), y-bond to (i, j + 1)."""
        n, L, N = len(v), self.L, self.L ** 2
        M = np.zeros((n, N, N))
        eta = (2.0 * v - 1.0).reshape(n, N).cpu().numpy()
        b = np.arange(N)
        i, j = b // L, b % L
        M[:, b, b] += 2.0 * eta
        M[:, b, (i + 1) % L * L + j] += 2.0
        c = b[j + 1 < L] if self.open else b
        M[:, c, c // L * L + (c % L + 1) % L] += 2.0
        parts = np.array_split(M, max(1, min(64, n // 4)))
        with ThreadPoolExecutor(os.cpu_count() or 4) as ex:
            s = np.concatenate(list(ex.map(lambda m: np.linalg.svd(m, compute_uv=False), parts)))
        return torch.as_tensor(s, device=DEV)

    @staticmethod
    def thermal(eps, beta):
        x = 0.5 * beta[:, None] * eps
        q = torch.exp(-2.0 * x)
        return ((x + torch.log1p(q)).sum(1), -(0.5 * eps * torch.tanh(x)).sum(1),
                (x * x * 4.0 * q / (1.0 + q) ** 2).sum(1))

    def evaluate(self, v):
        n, L = len(v), self.L
        F = -self.vb * v.sum((1, 2))
        for f in range(self.K):
            x = self.pre(v, f)
            F -= torch.logaddexp(x, torch.zeros_like(x)).sum((1, 2))
        d = dict(F=F, v=v)
        if self.kitaev:
            d["eps"] = self.spectrum(v)
            d["lp"], d["E"], cf = self.thermal(d["eps"], self.beta)
            flux = (v != v.roll((1, -1), (1, 2))).double()         # hexagon of cell r: z-bonds r and r - e1 + e2
            vison = flux[:, :, :L - 1].mean((1, 2)) if self.open else flux.mean((1, 2))
            d["obs"] = torch.stack([d["E"], d["E"] ** 2, cf, vison], 1)
        else:
            s = 2.0 * v - 1.0
            d["E"] = -(s * (s.roll(-1, 1) + s.roll(-1, 2))).sum((1, 2))
            d["lp"], m = -self.beta * d["E"], s.sum((1, 2))
            d["obs"] = torch.stack([d["E"], d["E"] ** 2, m.abs(), m ** 2], 1)
        return d

    @staticmethod
    def choose(yes, a, b):
        return {k: torch.where(yes.view(-1, *[1] * (a[k].dim() - 1)), a[k], b[k]) for k in a}

    def propose(self):
        new, old = self.evaluate(self.gibbs(1)), self.now
        logr = (new["lp"] - old["lp"]) + (new["F"] - old["F"])
        yes = _log_uniform(TAG_ACCEPT, self.step, self.cid, self.seed) < logr
        self.now = self.choose(yes, new, old)
        self.v = self.now["v"]
        self.acc += yes
        self.sums += self.now["obs"]
        self.step += 1

    def exchange(self):
        """Neighbouring temperatures: pairs (i, i + 1), i even on even steps and odd on odd ones."""
        n, par = len(self.v), self.step % 2
        i = torch.arange(par, n - 1, 2, device=DEV)
        if len(i):
            d, b = self.now, self.beta

            def at(x, y):                          # log pi_x of the lattice in slot y
                return self.thermal(d["eps"][y], b[x])[0] if self.kitaev else -b[x] * d["E"][y]
            logb = at(i, i + 1) + at(i + 1, i) - d["lp"][i] - d["lp"][i + 1]
            e = i[_log_uniform(TAG_TEMP, self.step, self.cid[i], self.seed) < logb]
            perm = torch.arange(n, device=DEV)
            perm[e], perm[e + 1] = e + 1, e
            d = {k: x[perm] for k, x in d.items()}
            if self.kitaev:
                d["lp"], d["E"], cf = self.thermal(d["eps"], b)
                d["obs"] = torch.stack([d["E"], d["E"] ** 2, cf, d["obs"][:, 3]], 1)
            else:
                d["lp"] = -b * d["E"]
            self.now, self.v = d, d["v"]

    def sweep(self, exchange):
        i = torch.arange(self.L, device=DEV)
        u = _uniform_plane(self.L, TAG_LOCAL, self.step, self.cid, self.seed)
        v = self.v
        for colour in (0, 1):
            s = 2.0 * v - 1.0
            dE = 2.0 * s * (s.roll(1, 1) + s.roll(-1, 1) + s.roll(1, 2) + s.roll(-1, 2))
            flip = (u < torch.exp(-self.beta[:, None, None] * dE)) & ((i[:, None] + i) % 2 == colour)
            v = torch.where(flip, 1.0 - v, v)
            self.acc += flip.sum((1, 2))
        self.v = v
        self.now = self.evaluate(v)
        if exchange:
            self.exchange()
        self.sums += self.now["obs"]
        self.step += 1
        return self.now["E"].clone()

    def result(self, energies=False):
        out = {"bits": _pack(self.v.to(torch.uint8)).view(np.int32), "sums": self.sums, "accepts": self.acc}
        if energies:
            out["logpi"], out["F"], out["E"] = self.now["lp"], self.now["F"], self.now["E"]
        return out


def _exact_autocorr(x):
    x = x.cpu().numpy()
    n = len(x)
    d = x - x.mean(0)
    g0 = (d * d).mean(0)
    tau, win = np.full(x.shape[1], 0.5), np.full(x.shape[1], n - 1, dtype=np.int64)
    live = np.arange(x.shape[1])
    for lag in range(1, n):
        tau[live] += (d[:n - lag, live] * d[lag:, live]).sum(0) / n / g0[live]
        done = lag >= 5.0 * tau[live]
        win[live[done]] = lag
        live = live[~done]
        if not len(live):
            break
    return [tau, win]


def _exact_train(case, seed):
    vs, ts, orders, thetas = _training_set(case, seed)
    K, k, L, n, P = (case[x] for x in ("K", "k", "L", "samples", "problems"))
    v, t = torch.stack(vs).double(), torch.stack(ts)
    order, th = torch.stack(orders).long(), torch.stack(thetas)
    m, s = torch.zeros_like(th), torch.zeros_like(th)
    i = torch.arange(L, device=DEV)
    taps = [((i[:, None] + a) % L * L + (i + b) % L).reshape(-1) for a in range(k) for b in range(k)]
    taps = torch.stack(taps)                                       # (k*k, N): site of tap ab of hidden unit n
    row = torch.arange(P, device=DEV)[:, None]
    losses = []
    for step, b0 in enumerate(range(0, n, BATCH), 1):
        o = order[:, b0:b0 + BATCH]
        x, M = v[row, o].reshape(P, -1, L * L), o.shape[1]
        win = x[:, :, taps]                                        # (P, M, k*k, N)
        W, vb, hb = th[:, :K * k * k].view(P, K, k * k), th[:, K * k * k], th[:, K * k * k + 1:]
        a = torch.einsum("pmcn,pfc->pmfn", win, W) + hb[:, None, :, None]
        F = -vb[:, None] * x.sum(2) - torch.logaddexp(a, torch.zeros_like(a)).sum((2, 3))
        diff = t[row, o] - F
        d = diff - diff.mean(1, keepdim=True)
        losses.append((d * d).mean(1))
        sig, w = torch.sigmoid(a), 2.0 / M * d
        gW = torch.einsum("pm,pmfn,pmcn->pfc", w, sig, win).reshape(P, -1)
        gr = torch.cat([gW, torch.einsum("pm,pm->p", w, x.sum(2))[:, None], torch.einsum("pm,pmf->pf", w, sig.sum(3))], 1)
        m, s = B1 * m + (1.0 - B1) * gr, B2 * s + (1.0 - B2) * gr * gr
        th = th - LR * (m / (1.0 - B1 ** step)) / (torch.sqrt(s / (1.0 - B2 ** step)) + EPS)
    return {"theta": th, "m": m, "v": s, "t": torch.full((P, 1), step, dtype=torch.int64), "losses": torch.stack(losses, 1)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "autocorr":
        return _exact_autocorr(_series(case, seed))
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "sweeps":
        n, L = case["chains"], case["L"]
        T = _ladder(case, n)
        c = Chains(ISING, np.zeros((1, 2, 2)), 0.0, np.zeros(1), _ising_lattices(n, L, T, seed, 1), T, int(seed), 0)
        trace = [c.sweep(case["exchange"]) for _ in range(case["S"])]
        return {**c.result(), "trace": torch.stack(trace)}
    W, vb, hb = _filters(case, seed)
    n = case["chains"]
    T = _ladder(case, n)
    if kind == "tempering":
        model = ISING if case["model"] == "ising" else KITAEV
        x, y = (Chains(model, W, vb, hb, _lattices(case, n, case["L"], T, seed, 1 + i), T, int(seed) + i, i * n)
                for i in (0, 1))
        for _ in range(case["S"]):
            new, old = y.evaluate(y.gibbs(case["g"])), x.now
            loga = (new["lp"] - old["lp"]) + (new["F"] - old["F"])
            yes = _log_uniform(TAG_SWAP, x.step, x.cid, x.seed) < loga
            x.now, y.now = x.choose(yes, new, old), x.choose(yes, old, new)
            x.acc += yes
            x.exchange()
            x.v, y.v = x.now["v"], y.now["v"]
            x.sums += x.now["obs"]
            x.step, y.step = x.step + 1, y.step + 1
        return {"phys": x.result(energies=True), "rbm": _pack(y.v.to(torch.uint8)).view(np.int32)}
    out = []
    for i, L in enumerate(_sides(case) if "Ls" in case else [case["L"]]):
        c = Chains(ISING if kind == "ising" else KITAEV, W, vb, hb, _lattices(case, n, L, T, seed, 1 + i), T, int(seed),
                   i * n)
        for _ in range(case["S"]):
            c.propose()
        out.append(c.result(energies=kind == "open" or (len(_sides(case)) == 1 and case["prec"] == "fp64")))
    if kind == "ising" and len(out) > 1:
        return {"bits": [r["bits"] for r in out], "sums": [r["sums"] for r in out]}
    return out if len(out) > 1 else out[0]
