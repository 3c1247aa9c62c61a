"""The network's tensor-core kernels when their bounded waits give up: every call reports the
time-out and ends, and with the default bound again the same handle gives the same bits as
before.  A negative bound makes the part that issues the products give up on its first operands,
with copies in flight and the epilogue waiting; the other roles give up after its absolute value."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MGMC_ERR_TIMEOUT = 5


# whole-line kernels (side >= 128), per-tap kernels, weight gradients; c0 = 8: the im2col products
@pytest.mark.parametrize("n,c0,batch", [(255, 32, 2), (127, 16, 3), (63, 32, 2), (31, 8, 1)])
def test_give_up_is_reported_and_the_handle_recovers(n, c0, batch):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import MGMCError, Unet
    build.build()
    g = torch.Generator(device="cuda").manual_seed(n + c0)
    x = torch.randn(batch, n + 1, n + 1, 3, generator=g, device="cuda").bfloat16()
    t = torch.randn(batch, n * n, generator=g, device="cuda")
    net = Unet(n, c0=c0, max_batch=batch, seed=3)
    y0 = net.predict(x)
    loss0, g0 = net.gradient(x, t, batch)
    for limit in (-500_000, -1):
        net.set_wait_limit(limit)
        for call in (lambda: net.predict(x), lambda: net.gradient(x, t, batch)):
            with pytest.raises(MGMCError) as e:
                call()
            assert e.value.code == MGMC_ERR_TIMEOUT
    net.set_wait_limit(0)
    assert torch.equal(net.predict(x), y0)
    loss1, g1 = net.gradient(x, t, batch)
    assert loss1 == loss0 and np.array_equal(g1, g0)
    net.close()
