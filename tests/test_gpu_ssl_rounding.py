"""Rounding error of the squared operator's W-cycle on the GPU against the same cycle in extended
precision (numpy's long double, written from the definitions): no observations and kappa^2 = 16 on
31^2, where every operator entry is exact in FP64, so that the difference is the sampler's rounding
alone.  The one-CTA kernel of the small grids sums a residual in another order than the
one-launch-per-phase kernels; its states may have at most 1.7 times their rounding error (rms over
chains; the orders have the same bounds, 1.7 allows for the scatter of six chains -- a residual
that begins with the centre's product has 3.5 times)."""
import numpy as np
import pytest

from paper_2407_12149_gb300 import inputs

pytestmark = pytest.mark.gpu

LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")
N, K2, CYCLES, SEEDS = 31, 16, 3, range(6)


def _philox(c0, cycle, w3, seed):
    u, m = np.uint64, 0xFFFFFFFF
    k0, k1 = seed & m, seed >> 32
    c = [c0.astype(u)] + [np.full_like(c0, v).astype(u) for v in (cycle, 0, w3)]
    for _ in range(10):
        p0, p1 = c[0] * u(0xD2511F53), c[2] * u(0xCD9E8D57)
        c = [(p1 >> u(32)) ^ c[1] ^ u(k0), p1 & u(m), (p0 >> u(32)) ^ c[3] ^ u(k1), p0 & u(m)]
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c


def _box_muller(u1, u2):
    r = np.sqrt(LD(-2) * np.log(u1))
    return r * np.cos(2 * PI * u2), r * np.sin(2 * PI * u2)


def _site_normals(seed, n, cycle, level, slot):
    nq = (n + 3) // 4
    u = [(v.astype(LD) + LD(0.5)) * LD(2) ** -32 for v in _philox(np.arange(n * nq), cycle, (level << 16) | slot, seed)]
    (a0, a1), (b0, b1) = _box_muller(u[0], u[1]), _box_muller(u[2], u[3])
    return np.stack([a0, b0, a1, b1], 1).reshape(n, 4 * nq)[:, :n]


def _coarsest_normal(seed, cycle, slot):
    w = [int(v[0]) for v in _philox(np.arange(1), cycle, (2 << 24) | slot, seed)]
    k = [(w[0] << 21) | (w[1] >> 11), (w[2] << 21) | (w[3] >> 11)]
    return _box_muller(*[(LD(v) + LD(0.5)) * LD(2) ** -53 for v in k])[0]


def _prolong(c):
    for _ in range(2):   # one axis, then the other
        f = np.zeros((2 * c.shape[0] + 1, c.shape[1]), LD)
        f[1::2] = c
        f[0:-1:2] += c / 2
        f[2::2] += c / 2
        c = f.T
    return c


def _restrict(f):
    for _ in range(2):
        f = (f[1::2] + (f[0:-1:2] + f[2::2]) / 2).T
    return f


class _Grid:
    def __init__(self, n, coef):
        self.n, self.coef, self.diag = n, coef, coef[12]
        j, i = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
        self.colours = [(i % 3) + 3 * (j % 3) == c for c in range(9)]
        self.used = [o for o in range(25) if (coef[o] != 0).any()]

    def apply(self, x):
        xp, out = np.pad(x, 2), np.zeros_like(x)
        for o in self.used:
            out += self.coef[o] * xp[o // 5:o // 5 + self.n, o % 5:o % 5 + self.n]
        return out

    def sweep(self, x, f, colours):
        for c in colours:
            x = np.where(c, x + (f - self.apply(x)) / self.diag, x)
        return x

    def coarser(self):
        nc = (self.n - 1) // 2
        coef = np.zeros((25, nc, nc), LD)
        j, i = np.meshgrid(np.arange(nc), np.arange(nc), indexing="ij")
        for p in range(25):
            w = _restrict(self.apply(_prolong(((i % 5 == p % 5) & (j % 5 == p // 5)).astype(LD))))
            for o in range(25):
                hit = ((i + o % 5 - 2) % 5 == p % 5) & ((j + o // 5 - 2) % 5 == p // 5)
                coef[o] = np.where(hit, w, coef[o])
        return _Grid(nc, coef)


def _hierarchy():
    h, k2 = LD(1) / (N + 1), LD(K2)
    coef = np.zeros((25, N, N), LD)
    sides = np.zeros((N, N), LD)
    for a in (0, -1):
        sides[a] += 1
        sides[:, a] += 1
    for o in range(25):
        d = sorted((abs(o % 5 - 2), abs(o // 5 - 2)))
        bih = {(0, 0): 20, (0, 1): -8, (1, 1): 2, (0, 2): 1}.get(tuple(d), 0)
        coef[o] = h * h * (LD(bih) / h ** 4 + 2 * k2 * LD({0: 4, 1: -1}.get(sum(d), 0)) / h ** 2)
    coef[12] += h * h * (sides / h ** 4 + k2 * k2)
    grids = [_Grid(N, coef)]
    while grids[0].n > 1:
        grids.insert(0, grids[0].coarser())
    return grids


def _chain(grids, seed):
    x = np.zeros((N, N), LD)

    def smooth(l, x, f, backward, slot, cycle):
        g = grids[l]
        return g.sweep(x, f + np.sqrt(g.diag) * _site_normals(seed, g.n, cycle, l, slot), g.colours[::-1] if backward else g.colours)

    def level(l, x, f, visit, cycle):
        v = visit[l]
        visit[l] += 1
        if l == 0:
            a = grids[0].diag
            return (f + np.sqrt(a) * _coarsest_normal(seed, cycle, v)) / a
        x = smooth(l, x, f, False, 2 * v, cycle)
        fc = _restrict(f - grids[l].apply(x))
        psi = np.zeros_like(fc)
        for _ in range(1 if l == len(grids) - 1 else 2):
            psi = level(l - 1, psi, fc, visit, cycle)
        return smooth(l, x + _prolong(psi), f, True, 2 * v + 1, cycle)

    for cycle in range(CYCLES):
        x = level(len(grids) - 1, x, np.zeros_like(x), [0] * len(grids), cycle)
    return x.ravel()


def test_rounding_error_of_the_one_cta_kernel():
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import Sampler
    build.build()
    if np.finfo(LD).nmant < 63:
        pytest.skip("no extended precision")
    grids = _hierarchy()
    p = inputs.make_problem("r", 2, N, kappa2_const=float(K2), m=0, disc=2, qoi_cells=4)
    err = {}
    for cmax in (1, 0):          # a launch per phase; one CTA
        s = Sampler(p, precision="fp64", coarse_max_n=cmax)
        got = []
        for seed in SEEDS:
            x = s.zeros()
            s.sample(x, CYCLES, 500 + seed)
            got.append(x.cpu().numpy())
        err[cmax] = np.stack(got)
        s.close()
    ref = np.stack([_chain(grids, 500 + seed) for seed in SEEDS])
    rms = {k: float(np.sqrt(np.mean((v - ref) ** 2) / np.mean(ref ** 2))) for k, v in err.items()}
    assert rms[1] <= 5e-14, rms   # the reference is the same chain: 100 roundings of 20 times the state
    assert rms[0] <= 1.7 * rms[1], rms
