"""plc_log_stats on fields with empty cells (1 + delta <= 0): alone, in runs
that fill a thread's four cells and in runs that do not, negative zeros, NaNs of
both signs; counts must be those of the cells one by one, and the moments those
of the others (1e-12: FP64 sums over at most 32^3 values within one ulp).
"""
import time

import numpy as np
import pytest
import torch

from tests.gpu_util import dev, ensure_lib

pytestmark = pytest.mark.gpu

N = 32


@pytest.mark.parametrize("run", [1, 3, 4, 5, 8, 64, 1000, N ** 3])
def test_counts_and_moments(run):
    rng = np.random.default_rng(run)
    delta = np.expm1(rng.standard_normal(N ** 3))
    empty = (np.arange(N ** 3) // run) % 2 == 0
    delta[empty] = -1.0 - rng.integers(0, 2, int(empty.sum()))
    bad = rng.choice(np.flatnonzero(empty), 40, replace=False)
    delta[bad[:20]] = np.nan
    delta[bad[20:]] = np.copysign(np.nan, -1.0)
    c = ensure_lib().Context(N, 100.0, "fp64")
    counts, outside, moments = c.log_stats(dev(delta.reshape(N, N, N), torch.float64), -6.0, 0.5, 24)
    u = 1.0 + delta[~empty]
    j = np.floor((np.log(u) + 6.0) / 0.5).clip(-1, 24).astype(int)
    want = np.bincount(j + 1, minlength=26)
    assert list(counts) == list(want[1:-1])
    assert list(outside) == [want[0], want[-1], int(empty.sum())]
    if u.size:
        x = np.log(u)
        d = x - x.mean()
        var = (d * d).mean()
        np.testing.assert_allclose(moments, [x.mean(), var, (d ** 3).mean() / var ** 1.5,
                                             (d ** 4).mean() / var ** 2 - 3.0], rtol=1e-12, atol=1e-12)


def test_empty_cells_cost_less_than_full_ones():
    # an empty field needs no logarithm: a third of a full one's time where it
    # takes none, the same where it does; the line lies between
    c = ensure_lib().Context(256, 100.0, "fp64")
    gen = torch.Generator(device="cuda").manual_seed(1)
    full = torch.expm1(torch.randn((256,) * 3, dtype=torch.float64, device="cuda", generator=gen))

    def best(delta):
        t = []
        for _ in range(20):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            c.log_stats(delta, -6.0, 0.05, 240)
            t.append(time.perf_counter() - t0)
        return min(t)
    assert best(torch.full_like(full, -1.0)) < 0.7 * best(full)
