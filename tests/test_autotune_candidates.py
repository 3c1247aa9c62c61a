"""The thread counts the autotuner times are launches of their own: none above the coarse kernel's
limit (512 threads in FP32, 256 in FP64), where the kernel would run at the limit again."""
import pytest

from paper_2407_12149_gb300 import autotune


class _Sampler:
    def __init__(self):
        self.band = self.threads = 0

    def set_band_min_n(self, v):
        self.band = v

    def set_coarse_threads(self, v):
        self.threads = v

    def close(self):
        pass


class _P:
    n, dim = 127, 2


@pytest.mark.parametrize("precision,limit", [("fp32", 512), ("fp64", 256)])
def test_no_two_candidates_run_the_same_launch(precision, limit):
    timed = []

    def timer(s):
        timed.append((s.band, s.threads))
        return 1.0

    autotune.autotune([_P()], precision, make_sampler=lambda ps, c: _Sampler(), timer=timer)
    threads = [t for _, t in timed[len(autotune.band_candidates([_P()], 31)):]]
    assert len(set(min(t, limit) for t in threads)) == len(threads) and max(threads) == limit
