"""A caller's allocator that aligns to 8 bytes only: the handles align within its blocks, give every
block back, and compute the bits they compute on torch's blocks."""
import numpy as np
import pytest

from paper_2407_12149_gb300 import inputs

pytestmark = pytest.mark.gpu


class _Shifted:
    """mgmc_allocator whose blocks start 8 bytes into torch's (aligned) ones."""

    live = None

    def __init__(self, device=0):
        import torch
        from paper_2407_12149_gb300 import mgmc
        _Shifted.live = live = set()

        def alloc(nbytes, stream, ctx):
            p = torch.cuda.caching_allocator_alloc(int(nbytes) + 8, device) + 8
            live.add(p)
            return p

        def free(ptr, stream, ctx):
            live.remove(ptr)
            torch.cuda.caching_allocator_delete(ptr - 8)

        self._a, self._f = mgmc.ALLOC_FN(alloc), mgmc.FREE_FN(free)
        self.struct = mgmc.mgmc_allocator(self._a, self._f, None)


@pytest.fixture
def shifted(monkeypatch):
    from paper_2407_12149_gb300 import build, mgmc
    build.build()
    plain = mgmc.TorchAllocator

    def use(on):
        monkeypatch.setattr(mgmc, "TorchAllocator", _Shifted if on else plain)
    return use


# one CTA for all grids, streamed and tiled grids, the W-cycle, Gibbs, 3D
@pytest.mark.parametrize("dim,n,precision,kw", [(2, 31, "fp64", {}), (2, 255, "fp32", {}), (2, 127, "fp64", {}),
                                                (2, 127, "fp32", dict(gamma=2)), (2, 63, "fp32", dict(gibbs=True)),
                                                (3, 31, "fp32", {})])
def test_sampler(shifted, dim, n, precision, kw):
    import torch
    from paper_2407_12149_gb300.mgmc import Sampler
    p = inputs.make_problem("a", dim, n, kappa2_seed=3, m=5, obs_seed=4, qoi_cells=8)
    got = []
    for on in (False, True):
        shifted(on)
        s = Sampler(p, precision=precision, **kw)
        x = s.zeros()
        s.sample(x, 3, 9)
        s.check_status()
        got.append(x)
        s.close()
    assert torch.equal(got[0], got[1]) and not _Shifted.live


def test_unet(shifted):
    import torch
    from paper_2407_12149_gb300.mgmc import Unet
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(2, 128, 128, 3, generator=g, device="cuda").bfloat16()
    t = torch.randn(2, 127 * 127, generator=g, device="cuda")
    got = []
    for on in (False, True):
        shifted(on)
        net = Unet(127, c0=16, max_batch=2, seed=3)
        got.append((net.predict(x), net.gradient(x, t, 2)))
        net.close()
    assert torch.equal(got[0][0], got[1][0]) and np.array_equal(got[0][1][1], got[1][1][1]) and not _Shifted.live
