"""Performance cases of the sampler: what a program that uses this library has it do.

Every case goes through the public entry points (Sampler, BatchSampler, Unet, tc_gemm) on
device buffers.  exact() evaluates the same computation in FP64 with plain torch / numpy,
written from the definitions: the posterior hierarchy from its stencils, the Philox noise
streams, the V- or W-cycle of the low-rank Gibbs smoother, the U-Net as torch convolutions.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2407_12149_gb300 import inputs, mgmc

DEV = "cuda:0"
FD, Q1, SSL = 0, 1, 2


def _chain(name, n, precision, steps, **kw):
    c = dict(name=name, kind="chain", dim=2, n=n, coarsest=1, precision=precision, steps=steps, m=16, disc=FD,
             vary=True, gibbs=False, gamma=0, nu1=1, nu2=1)
    c.update(kw)
    return c


def listed():
    return [
        # smallest chain of the paper's tables (31^2, four grids, no observations): launch and
        # latency bound, the call a convergence study makes thousands of times
        _chain("chain-2d-31-fp64", 31, "fp64", 8, m=0, vary=False, coarsest=3),
        # one posterior chain of middling size in the fast precision
        _chain("chain-2d-255-fp32", 255, "fp32", 4),
        # the same posterior at the benchmark's resolution in full precision (the reference
        # chain that the batched FP32 chains are checked against)
        _chain("chain-2d-1023-fp64", 1023, "fp64", 2),
        # one 3D posterior chain (32 observations, coarsest grid 3^3)
        _chain("chain-3d-127-fp32", 127, "fp32", 2, dim=3, coarsest=3, m=32, vary=False),
        # the squared shifted Laplacian (13-point stencil) with the W-cycle of Table 1c
        _chain("wcycle-ssl-255-fp64", 255, "fp64", 1, disc=SSL, vary=False, m=8),
        # the plain Gibbs sampler that the paper compares against (Table 1a: Q1 elements)
        _chain("gibbs-q1-255-fp32", 255, "fp32", 8, disc=Q1, vary=False, m=8, gibbs=True),
        # the headline: independent chains of the 1023^2 posterior advanced together (one of
        # the benchmark's handles of eight chains)
        dict(name="batch8-2d-1023-fp32", kind="batch", sizes="1023", each=8, precision="fp32", steps=4, m=16),
        # chains of several resolutions in one handle
        dict(name="batch32-2d-mixed-fp32", kind="batch", sizes="63,127,255,511", each=8, precision="fp32", steps=4,
             m=16),
        # posterior mean by noise-free V-cycles: the targets of the learned warm start
        dict(name="mean-2d-255-fp64", kind="mean", dim=2, n=255, coarsest=1, precision="fp64", m=16, disc=FD,
             vary=True, gibbs=False, gamma=0, nu1=1, nu2=1, rtol=1e-8),
        # one training step's loss and gradient of the warm-start network (batch 8, 32 channels)
        dict(name="unet-gradient-255", kind="unet-gradient", n=255, c0=32, batch=8),
        # warm starts of a set of problems
        dict(name="unet-predict-255", kind="unet-predict", n=255, c0=32, batch=16),
        # the network's bottom convolution as a product (64 samples): bias, ReLU, BF16 output
        dict(name="gemm-65536x256x2304", kind="gemm", M=65536, N=256, K=2304, splits=1, bias=True, relu=True,
             bf16=True),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(["chain", "chain", "chain3", "wcycle", "gibbs", "batch", "batch", "mean", "unet-gradient",
                       "unet-predict", "gemm"])
    m = rng.choice([0, 1, 5, 8, 13, 16, 21, 32, 37])
    precision = rng.choice(["fp32", "fp64"])
    if kind == "chain":
        n = rng.choice([15, 31, 63, 127, 255, 511])
        disc = rng.choice([FD, FD, Q1])
        nu = rng.choice([(1, 1), (1, 1), (1, 1), (2, 1)])
        c = _chain("", n, precision, rng.randint(1, 5), m=m, disc=disc, vary=disc == FD, coarsest=rng.choice([1, 3, 7]),
                   nu1=nu[0], nu2=nu[1])
    elif kind == "chain3":
        c = _chain("", rng.choice([15, 31, 63]), precision, rng.randint(1, 4), dim=3, coarsest=rng.choice([1, 3]),
                   m=m, vary=rng.random() < 0.5)
    elif kind == "wcycle":
        disc = rng.choice([SSL, SSL, FD])
        c = _chain("", rng.choice([31, 63, 127, 255]), "fp64" if disc == SSL else precision, 1, m=m, disc=disc,
                   vary=disc == FD, gamma=2)
    elif kind == "gibbs":
        disc = rng.choice([FD, Q1])
        c = _chain("", rng.choice([31, 63, 127, 255, 511]), precision, rng.randint(1, 8), m=m, disc=disc,
                   vary=disc == FD, gibbs=True)
    elif kind == "batch":
        sizes = rng.sample([31, 63, 127, 255, 511], rng.randint(1, 3))
        most = max(1, min(16, 8 * 511 * 511 // sum(s * s for s in sizes)))
        c = dict(kind="batch", sizes=",".join(str(s) for s in sizes), each=rng.randint(1, most),
                 precision=rng.choice(["fp32", "fp32", "fp64"]), steps=rng.randint(1, 4), m=m)
    elif kind == "mean":
        c = dict(kind="mean", dim=2, n=rng.choice([31, 63, 127, 255]), coarsest=1, precision="fp64", m=m, disc=FD,
                 vary=True, gibbs=False, gamma=0, nu1=1, nu2=1, rtol=1e-8)
    elif kind == "unet-gradient":
        c = dict(kind=kind, n=rng.choice([63, 127, 255]), c0=rng.choice([8, 16, 32]), batch=rng.randint(1, 8))
    elif kind == "unet-predict":
        c = dict(kind=kind, n=rng.choice([63, 127, 255]), c0=rng.choice([8, 16, 32]), batch=rng.randint(1, 16))
    else:
        bf16 = rng.random() < 0.5
        c = dict(kind="gemm", M=_log_int(rng, 64, 65536), N=_log_int(rng, 8, 512), K=_log_int(rng, 32, 2304),
                 splits=1 if bf16 else rng.choice([1, 1, 3]), bias=False, relu=False, bf16=bf16)
        if c["splits"] == 1:
            c["bias"], c["relu"] = rng.random() < 0.5, rng.random() < 0.5
    c.pop("name", None)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _problem(case, n, dim, seed):
    """The posterior of one chain: kappa^2 field, observations and QoI from the seed."""
    m = case["m"]
    disc = case.get("disc", FD)
    vary = case.get("vary", True)
    return inputs.make_problem("case", dim, n, coarsest=min(case.get("coarsest", 1), n),
                               kappa2_seed=seed if vary else None,
                               kappa2_const={2: {FD: 10.0, Q1: 100.0, SSL: 100.0}[disc], 3: 25.0}[dim], m=m,
                               obs_seed=seed + 1, disc=disc, sigma2=1e-4 if disc == FD else 1.5e-6,
                               qoi_cells=max(2, (n + 1) // 8))


def _smooth(n, dim, seed, count=1):
    """`count` smooth fields of unit size on the n^dim interior vertices (FP64, device)."""
    rng = np.random.default_rng(seed)
    x = torch.linspace(1, n, n, dtype=torch.float64, device=DEV) / (n + 1)
    S = torch.stack([torch.sin(math.pi * k * x) for k in range(1, 9)])
    decay = 1.0 / np.add.outer(np.arange(1, 9) ** 2, np.arange(1, 9) ** 2)
    if dim == 3:
        decay = 1.0 / np.add.outer(1.0 / decay, np.arange(1, 9) ** 2)
    c = torch.tensor(rng.normal(size=(count,) + decay.shape) * decay, device=DEV)
    f = torch.einsum("bkl,ki,lj->bij", c, S, S) if dim == 2 else torch.einsum("bklm,ki,lj,mh->bijh", c, S, S, S)
    return f.reshape(count, -1)


def _problems(case, seed):
    if case["kind"] == "batch":
        ns = [int(s) for s in case["sizes"].split(",") for _ in range(case["each"])]
        return [_problem(case, n, 2, 7000 * seed + 10 * c) for c, n in enumerate(ns)]
    return [_problem(case, case["n"], case["dim"], 7000 * seed)]


def _start(case, problems, seed):
    """Initial states, one flat tensor (chain after chain)."""
    dt = torch.float32 if case["precision"] == "fp32" else torch.float64
    return torch.cat([_smooth(p.n, p.dim, 31 * seed + c)[0] for c, p in enumerate(problems)]).to(dt)


def _unet_params(c0, seed):
    """Flat parameters: He-normal 3x3 weights [cout][3][3][cin], small biases, a 1x1 output."""
    rng = np.random.default_rng(seed)
    parts = []
    for _, cin, cout in _unet_layers(c0):
        parts.append(rng.normal(0.0, math.sqrt(2.0 / (9 * cin)), cout * 9 * cin))
        parts.append(rng.normal(0.0, 0.02, cout))
    parts.append(rng.normal(0.0, math.sqrt(1.0 / c0), c0))
    parts.append(rng.normal(0.0, 0.02, 1))
    return np.concatenate(parts).astype(np.float32)


def _unet_data(case, seed):
    """Input channels (log kappa^2 / 10, observation weights, weighted data) and targets."""
    n, B = case["n"], case["batch"]
    x = torch.zeros(B, n + 1, n + 1, 3, dtype=torch.float64, device=DEV)
    x[:, :n, :n, 0] = 2.0 * _smooth(n, 2, seed + 5, B).view(B, n, n)
    for b in range(B):
        site, w = inputs.point_obs_rows(n, 2, inputs.obs_locations(16, 2, seed + b))
        y = inputs.obs_values(16, seed + b)
        for k in range(16):
            for s, v in zip(site[k], w[k]):
                if s >= 0:
                    x[b, int(s) // n, int(s) % n, 1] += float(v)
                    x[b, int(s) // n, int(s) % n, 2] += float(v) * float(y[k])
    return x.to(torch.bfloat16).contiguous(), (2.0 * _smooth(n, 2, seed + 6, B)).float().contiguous()


def _gemm_data(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    ld = (case["K"] + 7) // 8 * 8
    A = torch.relu(torch.randn(case["M"], ld, generator=g, device=DEV)).bfloat16()[:, :case["K"]]
    B = (torch.randn(case["N"], ld, generator=g, device=DEV) * math.sqrt(2.0 / case["K"])).bfloat16()[:, :case["K"]]
    bias = torch.randn(case["N"], generator=g, device=DEV) * 0.1 if case["bias"] else None
    return A, B, bias


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind.startswith("unet"):
        s["net"] = mgmc.Unet(case["n"], c0=case["c0"], max_batch=case["batch"], seed=seed)
        s["net"].set_params(_unet_params(case["c0"], seed))
        s["x"], s["t"] = _unet_data(case, seed)
    elif kind == "gemm":
        s["A"], s["B"], s["bias"] = _gemm_data(case, seed)
        s["epi"] = ((mgmc.EPI_BIAS if case["bias"] else 0) | (mgmc.EPI_RELU if case["relu"] else 0) |
                    (mgmc.EPI_BF16 if case["bf16"] else 0))
    else:
        ps = _problems(case, seed)
        s["x"] = _start(case, ps, seed)
        s["seed"], s["step"] = 1000 + seed, 0
        if kind == "batch":
            s["handle"] = mgmc.BatchSampler(ps, precision=case["precision"])
            s["xs"] = list(torch.split(s["x"], [p.N for p in ps]))
            s["qoi"] = torch.zeros(len(ps), case["steps"], dtype=torch.float64, device=DEV)
        else:
            s["handle"] = mgmc.Sampler(ps[0], precision=case["precision"], nu1=case["nu1"], nu2=case["nu2"],
                                       gibbs=case["gibbs"], gamma=case["gamma"])
            if kind == "chain":
                s["qoi"] = torch.zeros(case["steps"], dtype=torch.float64, device=DEV)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("chain", "batch"):
        x = s["x"] if kind == "chain" else s["xs"]
        s["handle"].sample(x, case["steps"], s["seed"], step_offset=s["step"], qoi=s["qoi"])
        s["step"] += case["steps"]
        # the series keeps the chain's own precision: the QoI of an FP32 state has no more
        return {"x": s["x"], "qoi": s["qoi"].to(s["x"].dtype)}
    if kind == "mean":
        x = torch.zeros_like(s["x"])
        cycles, _ = s["handle"].mean_solve(x, rtol=case["rtol"], max_cycles=100)
        return {"x": x, "cycles": cycles}
    if kind == "unet-gradient":
        loss, grad = s["net"].gradient(s["x"], s["t"], case["batch"])
        return {"loss": np.float32(loss), "grad": grad}
    if kind == "unet-predict":
        return s["net"].predict(s["x"])
    return mgmc.tc_gemm(s["A"], s["B"], splits=case["splits"], epilogue=s["epi"], bias=s["bias"])


def work(case):
    """Bytes and operations of one pass: each input read once, each output written once, the
    arithmetic of the method (two sweeps, a residual and the transfers of each grid, the
    Box-Muller normals counted as 40 operations a site and sweep)."""
    kind = case["kind"]
    if kind.startswith("unet"):
        H, B = case["n"] + 1, case["batch"]
        macs = sum(9 * ci * co * (H >> lv) ** 2 for lv, ci, co in _unet_layers(case["c0"])) + case["c0"] * H * H
        params = sum(9 * ci * co + co for _, ci, co in _unet_layers(case["c0"])) + case["c0"] + 1
        grad = kind == "unet-gradient"
        return {"bytes": B * (6 * H * H + 4 * case["n"] ** 2) + params * (8 if grad else 4),
                "flops": (6 if grad else 2) * macs * B}
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 2 * (M * K + N * K) + (2 if case["bf16"] else 4) * M * N, "flops": 2 * M * N * K}
    elem = 4 if case["precision"] == "fp32" else 8
    ns = [int(v) for v in case["sizes"].split(",")] * case["each"] if kind == "batch" else [case["n"]]
    dim = case.get("dim", 2)
    steps = case.get("steps", 10)
    sites = sum(n ** dim for n in ns)
    disc = case.get("disc", FD)
    nnz = {FD: 2 * dim + 1, Q1: 3 ** dim, SSL: 25}[disc]
    sweeps = case.get("nu1", 1) + case.get("nu2", 1)
    # coarser grids: all visits of the V-cycle add 1 / (2^dim - 1) of the finest grid's sites, those
    # of the W-cycle 1 / (2^dim - 2); their stencils have 3^dim (SSL: 25) entries
    wcycle = case.get("gamma", 0) == 2 or disc == SSL
    cfrac = 0.0 if case.get("gibbs") else 1.0 / (2 ** dim - (2 if wcycle else 1))
    cnnz = 25 if disc == SSL else 3 ** dim
    noise = 0 if kind == "mean" else 40
    per = sweeps * (2 * nnz + noise) + (0 if case.get("gibbs") else 2 * nnz)
    perc = cfrac * (sweeps * (2 * cnnz + noise) + 2 * cnnz)
    # per cycle: the state read and written, the operator (one value a site of the finite-difference
    # finest grid, the symmetric half of the others) read
    coefs = (1 if disc == FD else (nnz + 1) // 2) + cfrac * (cnnz + 1) // 2
    return {"bytes": steps * sites * elem * (2 + coefs), "flops": steps * sites * (per + perc)}


# ---------------------------------------------------------------------------
# FP64 values from the definitions
# ---------------------------------------------------------------------------
M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 words (int64 tensors holding 32-bit values) of counters c0 (tensor), c1..c3."""
    k0, k1 = seed & M32, (seed >> 32) & M32
    c = [c0] + [torch.full_like(c0, v) for v in (c1, c2, c3)]
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & M32) ^ c[1] ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c[3] ^ k1, p0 & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _box_muller(u1, u2):
    r = torch.sqrt(-2.0 * torch.log(u1))
    return r * torch.cos(2.0 * math.pi * u2), r * torch.sin(2.0 * math.pi * u2)


class _Noise:
    """The random streams of one chain: counter (c0, cycle, chain, kind | level | slot)."""

    def __init__(self, seed, chain):
        self.seed, self.chain = seed, chain

    def words(self, c0, cycle, kind, level, slot):
        return _philox(c0, cycle & M32, ((cycle >> 32) & 0xFFFF) | (self.chain << 16),
                       (kind << 24) | (level << 16) | slot, self.seed)

    def site(self, n, dim, cycle, level, slot):
        nq = (n + 3) // 4
        rows = n ** (dim - 1)
        w = self.words(torch.arange(rows * nq, device=DEV), cycle, 0, level, slot)
        u = [(v.double() + 0.5) * 2.0 ** -32 for v in w]
        a0, a1 = _box_muller(u[0], u[1])
        b0, b1 = _box_muller(u[2], u[3])
        return torch.stack([a0, b0, a1, b1], 1).view(rows, 4 * nq)[:, :n].reshape((n,) * dim)

    def pairs(self, count, cycle, kind, level, slot):
        w = self.words(torch.arange((count + 1) // 2, device=DEV), cycle, kind, level, slot)
        u1 = (((w[0] << 21) | (w[1] >> 11)).double() + 0.5) * 2.0 ** -53
        u2 = (((w[2] << 21) | (w[3] >> 11)).double() + 0.5) * 2.0 ** -53
        return torch.stack(_box_muller(u1, u2), 1).reshape(-1)[:count]


def _along(x, axis, f):
    return f(x.movedim(axis, -1)).movedim(-1, axis)


def _prolong(x, dim):
    def one(c):
        f = c.new_zeros(c.shape[:-1] + (2 * c.shape[-1] + 1,))
        f[..., 1::2] = c
        f[..., 0:-1:2] += 0.5 * c
        f[..., 2::2] += 0.5 * c
        return f
    for a in range(-dim, 0):
        x = _along(x, a, one)
    return x


def _restrict(x, dim):
    for a in range(-dim, 0):
        x = _along(x, a, lambda f: f[..., 1::2] + 0.5 * (f[..., 0:-1:2] + f[..., 2::2]))
    return x


class _Grid:
    """One grid: stencil coefficients [W^dim, n, ...], observation columns, smoother data."""

    def __init__(self, dim, n, R, coef, B, Gamma):
        self.dim, self.n, self.R, self.W, self.coef, self.B = dim, n, R, 2 * R + 1, coef, B
        self.diag = coef[(self.W ** dim - 1) // 2]
        self.used = [o for o in range(self.W ** dim) if bool((coef[o] != 0).any())]
        ax = torch.arange(n, device=DEV)
        idx = [ax.view([-1 if k == a else 1 for k in range(dim)]) for a in range(dim)]   # (k, j, i)
        if R == 1:
            code = sum((idx[dim - 1 - a] % 2) << a for a in range(dim))
            seq = [0, 3, 2, 1] if dim == 2 else [0, 6, 5, 3, 4, 2, 1, 7]
        else:
            code, seq = idx[1] % 3 + 3 * (idx[0] % 3), list(range(9))
        self.colours = [code == c for c in seq]
        self.G = [None, None]
        if B is not None:
            for d in (0, 1):
                C = self.sweep(torch.zeros_like(B), B, d)
                S = Gamma + self.dot(C)
                self.G[d] = torch.einsum("k...,kl->l...", C, torch.linalg.inv(S))

    def dot(self, x):
        """B^T x (of a field, or of a stack of m fields)."""
        m = self.B.shape[0]
        b = self.B.reshape(m, -1)
        return b @ x.reshape(-1) if x.dim() == self.dim else b @ x.reshape(x.shape[0], -1).T

    def apply(self, x):
        xp = F.pad(x, (self.R,) * (2 * self.dim))
        out = torch.zeros_like(x)
        for o in self.used:
            s = [(o // self.W ** a) % self.W for a in range(self.dim - 1, -1, -1)]
            out.addcmul_(self.coef[o].expand_as(out), xp[(Ellipsis,) + tuple(slice(v, v + self.n) for v in s)])
        return out

    def sweep(self, x, f, direction):
        for c in (self.colours if direction == 0 else self.colours[::-1]):
            x = torch.where(c, x + (f - self.apply(x)) / self.diag, x)
        return x

    def coarser(self, Gamma):
        """Galerkin grid P^T A P, each stencil class probed with the unit vectors of a lattice."""
        nc, W, dim = (self.n - 1) // 2, self.W, self.dim
        coef = torch.zeros((W ** dim,) + (nc,) * dim, dtype=torch.float64, device=DEV)
        ax = torch.arange(nc, device=DEV)
        idx = [ax.view([-1 if k == a else 1 for k in range(dim)]) for a in range(dim)]
        for p in range(W ** dim):
            cls = [(p // W ** a) % W for a in range(dim - 1, -1, -1)]
            on = sum((idx[a] % W == cls[a]).long() for a in range(dim)) == dim
            w = _restrict(self.apply(_prolong(on.double(), dim)), dim)
            for o in range(W ** dim):
                s = [(o // W ** a) % W - self.R for a in range(dim - 1, -1, -1)]
                hit = sum(((idx[a] + s[a]) % W == cls[a]).long() for a in range(dim)) == dim
                coef[o] = torch.where(hit, w, coef[o])
        return _Grid(dim, nc, self.R, coef, None if self.B is None else _restrict(self.B, dim), Gamma)


class _Chain:
    """The hierarchy and the MGMC cycle of one posterior."""

    def __init__(self, p, case):
        dim, n = p.dim, p.n
        h = 1.0 / (n + 1)
        shape = (n,) * dim
        k2 = (torch.full(shape, float(p.kappa2_const), dtype=torch.float64, device=DEV) if p.kappa2 is None else
              torch.tensor(p.kappa2, device=DEV).view(shape))
        one = torch.ones(shape, dtype=torch.float64, device=DEV)
        R = 2 if p.disc == SSL else 1
        W = 2 * R + 1
        coef = torch.zeros((W ** dim,) + shape, dtype=torch.float64, device=DEV)
        mid = (W ** dim - 1) // 2
        if p.disc == FD:
            coef[mid] = h ** dim * (k2 + 2 * dim / h ** 2)
            for a in range(dim):
                coef[mid - 3 ** a] = coef[mid + 3 ** a] = -h ** (dim - 2) * one
        elif p.disc == Q1:
            for o in range(9):
                d = abs(o % 3 - 1) + abs(o // 3 - 1)
                coef[o] = (8.0 if d == 0 else -1.0) / 3.0 + k2 * h * h * (16.0, 4.0, 1.0)[d] / 36.0
        else:
            sides = torch.zeros(shape, dtype=torch.float64, device=DEV)
            for a in range(2):
                for e in (0, n - 1):
                    sides.select(a, e).add_(1.0)
            for o in range(25):
                dx, dy = abs(o % 5 - 2), abs(o // 5 - 2)
                bih = {(0, 0): 20.0, (1, 0): -8.0, (1, 1): 2.0, (2, 0): 1.0}.get((max(dx, dy), min(dx, dy)), 0.0)
                lap = {0: 4.0, 1: -1.0}.get(dx + dy, 0.0)
                coef[o] = h * h * (bih / h ** 4 + 2.0 * k2 * lap / h ** 2)
            coef[mid] += h * h * (sides / h ** 4 + k2 * k2)
        self.m, B, self.Gamma = p.m, None, None
        if p.m:
            B = torch.zeros(p.m, n ** dim, dtype=torch.float64)
            for k in range(p.m):
                for s, w in zip(p.obs_site[k], p.obs_w[k]):
                    if s >= 0:
                        B[k, int(s)] += float(w)
            B = B.to(DEV).view((p.m,) + shape)
            self.Gamma = torch.tensor(p.Gamma, device=DEV)
            self.Gi = torch.linalg.inv(self.Gamma)
            self.LG = torch.linalg.cholesky(self.Gamma)
            self.y = torch.tensor(p.y, device=DEV)
        self.grids = [_Grid(dim, n, R, coef, B, self.Gamma)]
        for _ in range(p.n_levels - 1):
            self.grids.insert(0, self.grids[0].coarser(self.Gamma))
        g0 = self.grids[0]
        n0 = g0.n ** dim
        A0 = g0.apply(torch.eye(n0, dtype=torch.float64, device=DEV).view((n0,) + (g0.n,) * dim)).reshape(n0, n0)
        if B is not None:
            b0 = g0.B.reshape(self.m, n0)
            A0 = A0 + b0.T @ self.Gi @ b0
        self.L0 = torch.linalg.cholesky(0.5 * (A0 + A0.T))
        self.p, self.dim = p, dim
        self.nu = (case.get("nu1", 1), case.get("nu2", 1))
        self.gibbs = case.get("gibbs", False)
        self.gamma = case.get("gamma", 0) or (2 if p.disc == SSL else 1)
        self.qs = torch.tensor(p.qoi_site, device=DEV).long()
        self.qw = torch.tensor(p.qoi_w, device=DEV)

    def smooth(self, l, x, f, d, direction, slot):
        g = self.grids[l]
        rhs = f
        if self.noise:
            rhs = f + torch.sqrt(g.diag) * self.noise.site(g.n, self.dim, self.cycle, l, slot)
        x = g.sweep(x, rhs, direction)
        if self.m:
            v = g.dot(x) - d
            if self.noise:
                v = v - self.LG @ self.noise.pairs(self.m, self.cycle, 1, l, slot)
            x = x - torch.einsum("k...,k->...", g.G[direction], v)
        return x

    def level(self, l, x, f, d, visit):
        g = self.grids[l]
        v = visit[l]
        visit[l] += 1
        if l == 0:
            r = f.reshape(-1)
            if self.m:
                r = r + (self.Gi @ d) @ g.B.reshape(self.m, -1)
            r = torch.linalg.solve_triangular(self.L0, r[:, None], upper=False)
            if self.noise:
                r = r + self.noise.pairs(r.shape[0], self.cycle, 2, 0, v)[:, None]
            return torch.linalg.solve_triangular(self.L0.T, r, upper=True).view_as(x)
        S = max(1, *self.nu)
        for j in range(self.nu[0]):
            x = self.smooth(l, x, f, d, 0, 2 * (v * S + j))
        if not self.gibbs:
            fc = _restrict(f - g.apply(x), self.dim)
            dc = d - g.dot(x) if self.m else d
            psi = torch.zeros_like(fc)
            for _ in range(1 if l == len(self.grids) - 1 else self.gamma):
                psi = self.level(l - 1, psi, fc, dc, visit)
            x = x + _prolong(psi, self.dim)
        for j in range(self.nu[1]):
            x = self.smooth(l, x, f, d, 1, 2 * (v * S + j) + 1)
        return x

    def steps(self, x, count, noise):
        """`count` cycles from x: the state and the QoI after each."""
        self.noise = noise
        top = self.grids[-1]
        x, q = x.double().view((top.n,) * self.dim), []
        f, d = torch.zeros_like(x), self.y if self.m else None
        for self.cycle in range(count):
            x = self.level(len(self.grids) - 1, x, f, d, [0] * len(self.grids))
            q.append((x.reshape(-1)[self.qs] * self.qw).sum())
        return x.reshape(-1), torch.stack(q)

    def mean(self, rtol):
        top = self.grids[-1]
        x = torch.zeros((top.n,) * self.dim, dtype=torch.float64, device=DEV)

        def rhs(v):
            return torch.einsum("k...,k->...", top.B, self.Gi @ v) if self.m else torch.zeros_like(x)
        norm = float(rhs(self.y).norm()) if self.m else 0.0
        cycles = 0

        def rel():
            r = float((rhs(self.y - top.dot(x)) - top.apply(x)).norm()) if self.m else float(top.apply(x).norm())
            return r / norm if norm > 0.0 else (0.0 if r == 0.0 else math.inf)
        while rel() > rtol and cycles < 100:
            for _ in range(min(1 if cycles < 4 else 2, 100 - cycles)):
                x = self.steps(x, 1, None)[0].view_as(x)
                cycles += 1
        return x.reshape(-1), cycles


def _unet_layers(c0):
    """(level, input channels, output channels) of the 14 convolutions."""
    c = [c0 << s for s in range(4)]
    return [(0, 3, c[0]), (0, c[0], c[0]), (1, c[0], c[1]), (1, c[1], c[1]), (2, c[1], c[2]), (2, c[2], c[2]),
            (3, c[2], c[3]), (3, c[3], c[3]), (2, c[3] + c[2], c[2]), (2, c[2], c[2]), (1, c[2] + c[1], c[1]),
            (1, c[1], c[1]), (0, c[1] + c[0], c[0]), (0, c[0], c[0])]


def _conv3(x, W, b):
    """3x3 convolution as nine products of shifted pixels (channels last)."""
    xp = F.pad(x, (0, 0, 1, 1, 1, 1))
    H = x.shape[1]
    return b + sum(xp[:, ky:ky + H, kx:kx + H] @ W[:, ky, kx].T for ky in range(3) for kx in range(3))


def _unet_forward(theta, c0, x):
    o, it = 0, iter(_unet_layers(c0))

    def take(count):
        nonlocal o
        o += count
        return theta[o - count:o]

    def two(x):
        for _ in range(2):
            _, ci, co = next(it)
            x = torch.relu(_conv3(x, take(co * 9 * ci).view(co, 3, 3, ci), take(co)))
        return x
    skips = []
    for _ in range(3):
        x = two(x)
        skips.append(x)
        x = 0.25 * (x[:, 0::2, 0::2] + x[:, 1::2, 0::2] + x[:, 0::2, 1::2] + x[:, 1::2, 1::2])
    x = two(x)
    for s in (2, 1, 0):
        up = x.repeat_interleave(2, 1).repeat_interleave(2, 2)
        x = two(torch.cat([up, skips[s]], -1))
    w = take(c0)
    return x @ w + take(1)


def exact(case, seed):
    kind = case["kind"]
    if kind.startswith("unet"):
        n, B = case["n"], case["batch"]
        x, t = _unet_data(case, seed)
        theta = torch.tensor(_unet_params(case["c0"], seed), device=DEV).double()
        if kind == "unet-predict":
            with torch.no_grad():
                return torch.cat([_unet_forward(theta, case["c0"], x[b:b + 1].double())[:, :n, :n].reshape(1, -1)
                                  for b in range(B)])
        theta.requires_grad_(True)
        loss, grad = 0.0, torch.zeros_like(theta)
        for b in range(B):
            e = _unet_forward(theta, case["c0"], x[b:b + 1].double())[:, :n, :n].reshape(-1) - t[b].double()
            part = (e * e).sum() / (B * n * n)
            grad += torch.autograd.grad(part, theta)[0]
            loss += float(part)
        return {"loss": np.float64(loss), "grad": grad.cpu().numpy()}
    if kind == "gemm":
        A, B, bias = _gemm_data(case, seed)
        C = A.double() @ B.double().T
        C = C if bias is None else C + bias.double()
        return torch.relu(C) if case["relu"] else C
    ps = _problems(case, seed)
    x0 = torch.split(_start(case, ps, seed), [p.N for p in ps])
    if kind == "mean":
        x, cycles = _Chain(ps[0], case).mean(case["rtol"])
        return {"x": x, "cycles": cycles}
    got = [_Chain(p, case).steps(x, case["steps"], _Noise(1000 + seed, c)) for c, (p, x) in enumerate(zip(ps, x0))]
    q = torch.stack([g[1] for g in got])
    return {"x": torch.cat([g[0] for g in got]), "qoi": q if kind == "batch" else q[0]}
