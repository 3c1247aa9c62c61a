"""Which sweeps a Gibbs handle runs, by its launches per step: two fused ones on FP32 9-point grids up
to 255^2, one per colour elsewhere (two colours on 5-point grids, four on 9-point ones), plus the
QoI launch and, with observations, two per low-rank step."""
import pytest

from paper_2407_12149_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,disc,n,sweeps", [("fp32", 1, 31, 2), ("fp32", 1, 255, 2), ("fp32", 1, 511, 8),
                                                     ("fp32", 0, 31, 4), ("fp32", 0, 511, 4), ("fp64", 1, 63, 8),
                                                     ("fp64", 0, 255, 4)])
@pytest.mark.parametrize("m", [0, 4])
def test_launches_per_step(precision, disc, n, sweeps, m):
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import Sampler
    build.build()
    p = inputs.make_problem("g", 2, n, kappa2_const=100.0, m=m, obs_seed=4, disc=disc, qoi_cells=4)
    s = Sampler(p, precision=precision, gibbs=True)
    assert s.launches_per_cycle() == sweeps + 1 + (4 if m else 0)
    s.close()
