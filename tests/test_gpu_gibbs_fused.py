"""The 2D Gibbs sampler with one sweep before and after (the V-cycle's fused sweep kernels)
and with two (one launch per colour) against the oracle, over both stencils, both
precisions and several sizes, with and without observations."""
import numpy as np
import pytest

import oracle
from paper_2407_12149_gb300 import inputs
from tests.test_gpu_parity import _check32, _check64, _run_gpu

pytestmark = pytest.mark.gpu


# sizes: the smallest grid with two levels, less than a tile, several tiles, the streamed FP32 range
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nu", [1, 2])
@pytest.mark.parametrize("n,m,disc", [(3, 1, 0), (7, 3, 1), (31, 0, 1), (127, 9, 0), (255, 16, 1), (511, 4, 0)])
def test_gibbs_matches_oracle(n, m, disc, nu, precision):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import Sampler
    build.build()
    p, xo, _ = _oracle(n, m, disc, nu)
    s = Sampler(p, precision=precision, gibbs=True, nu1=nu, nu2=nu)
    xg, qg = _run_gpu(torch, s, p, 5, 99)
    (_check64 if precision == "fp64" else _check32)(xg, xo)
    assert np.isfinite(qg).all()
    s.close()


def _oracle(n, m, disc, nu):
    p = inputs.make_problem("t", 2, n, n_levels=None, kappa2_seed=None if disc else 5, kappa2_const=100.0, m=m,
                            obs_seed=4, disc=disc, qoi_cells=(n + 1) // 4)
    o = oracle.Oracle(p.dim, p.n, p.n_levels, kappa2=p.kappa2, kappa2_const=p.kappa2_const, scale_hd=p.scale_hd,
                      disc=disc, nu1=nu, nu2=nu, obs_site=p.obs_site, obs_w=p.obs_w, Gamma=p.Gamma, y=p.y,
                      qoi_site=p.qoi_site, qoi_w=p.qoi_w)
    return (p, *o.sample(5, 99, gibbs=True))
