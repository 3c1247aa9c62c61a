"""The FP64 site normals, read back from a chain: one forward sweep from zero (Gibbs sampler,
no backward sweep) leaves sqrt(a_ii) z / a_ii at the sites of the first colour.  Compared with
numpy's FP64 evaluation of the same Philox words; the bound, 1e-15 of the largest radius, is five
roundings."""
import numpy as np
import pytest

from paper_2407_12149_gb300 import inputs

pytestmark = pytest.mark.gpu

M32 = np.uint64(0xFFFFFFFF)


def _philox(c0, c1, c2, c3, seed):
    k0, k1 = np.uint64(seed) & M32, (np.uint64(seed) >> np.uint64(32)) & M32
    c = [c0.astype(np.uint64)] + [np.full_like(c0, v, dtype=np.uint64) for v in (c1, c2, c3)]
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ k0, p1 & M32, (p0 >> np.uint64(32)) ^ c[3] ^ k1, p0 & M32]
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & M32, (k1 + np.uint64(0xBB67AE85)) & M32
    return c


@pytest.mark.parametrize("seed", [0, 7, (1 << 40) + 3])
def test_first_colour_of_a_sweep_is_the_scaled_normal(seed):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import Sampler
    build.build()
    n, k2 = 255, 10.0
    p = inputs.make_problem("n64", 2, n, kappa2_const=k2)
    s = Sampler(p, precision="fp64", nu1=1, nu2=0, gibbs=True)
    x = s.zeros()
    s.sample(x, 1, seed)
    x = x.cpu().numpy().reshape(n, n)
    h = 1.0 / (n + 1)
    a = h * h * (k2 + 4.0 / h ** 2)
    nq = (n + 3) // 4
    j = np.arange(n)
    w = _philox((j[:, None] * nq + np.arange(nq)[None, :]).ravel(), 0, 0, (p.n_levels - 1) << 16, seed)
    u = [(v.astype(np.float64) + 0.5) * 2.0 ** -32 for v in w]
    z = np.empty((n, 4 * nq))
    for off, (ua, ub) in ((0, (u[0], u[1])), (1, (u[2], u[3]))):
        r = np.sqrt(-2.0 * np.log(ua))
        z[:, off::4] = (r * np.cos(2.0 * np.pi * ub)).reshape(n, nq)
        z[:, off + 2::4] = (r * np.sin(2.0 * np.pi * ub)).reshape(n, nq)
    # red sites (i + j even) are updated first, from zero: x = sqrt(a) z / a
    red = (j[:, None] + j[None, :]) % 2 == 0
    ref = z[:, :n] / np.sqrt(a)
    assert np.abs(x - ref)[red].max() <= 1e-15 * 7.0 / np.sqrt(a)
    s.close()
