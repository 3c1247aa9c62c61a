"""Device memory of a network handle per sample of its batch: the activations, their gradients and
the buffers of the layers that still run as im2col products, nothing for the others."""
import pytest

pytestmark = pytest.mark.gpu


def _bytes_per_sample(n, c0):
    """What the handle's buffers take per sample (include/mgmc.h: layers and levels)."""
    c = [c0 << s for s in range(4)]
    layers = [(0, 3, c[0]), (0, c[0], c[0]), (1, c[0], c[1]), (1, c[1], c[1]), (2, c[1], c[2]), (2, c[2], c[2]),
              (3, c[2], c[3]), (3, c[3], c[3]), (2, c[3] + c[2], c[2]), (2, c[2], c[2]), (1, c[2] + c[1], c[1]),
              (1, c[1], c[1]), (0, c[1] + c[0], c[0]), (0, c[0], c[0])]
    P = [((n + 1) >> s) ** 2 for s in range(4)]
    col = [(P[s], -(-9 * ci // 8) * 8, co, l) for l, (s, ci, co) in enumerate(layers) if ci % 16 or co % 16]
    b = sum(6 * P[s] * co for s, ci, co in layers)                       # BF16 activation, FP32 gradient
    b += sum(2 * P[s + 1] * c[s] for s in range(3))                      # pooled
    b += sum(2 * P[s] * ci for l, (s, ci, co) in enumerate(layers) if l in (8, 10, 12))   # concatenated
    b += P[0] * (6 + 8) + 4 * n * n                                      # inputs, output and its gradient, targets
    b += 2 * max(P[s] * co for s, ci, co in layers)                      # dz
    b += 8 * max(P[s] * ci for s, ci, co in layers)                      # input gradients of a layer, twice
    b += 4 * max(p * k for p, k, co, l in col) + 2 * max(p * co for p, k, co, l in col)   # col, colT, dzT
    b += 4 * max([p * k for p, k, co, l in col if l > 0], default=0)     # dcol
    return b


@pytest.mark.parametrize("n,c0", [(127, 32), (127, 16), (63, 8)])
def test_memory_per_sample(n, c0):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import Unet
    build.build()

    def held(batch):
        before = torch.cuda.memory_allocated()
        net = Unet(n, c0=c0, max_batch=batch, seed=1)
        got = torch.cuda.memory_allocated() - before
        net.close()
        return got

    per = (held(24) - held(8)) / 16
    assert per <= 1.01 * _bytes_per_sample(n, c0), (per, _bytes_per_sample(n, c0))
