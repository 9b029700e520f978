"""The integer bin decisions of plc_log_stats against the FP64 expression
floor((ln(1 + delta) - lo) / width) they stand for, at bin widths, offsets and
values where the two could part: values on the edges and one ulp from them,
widths at and below the smallest the integer form takes, one bin, the most
bins, values near delta = 0 and beyond the logarithm's integer range.  Counts
are whole numbers and must agree exactly wherever the host's logarithm decides
the bin (farther from an edge than 4 ulp of it); the moments are FP64 sums of
values within one ulp: 1e-12 relative covers the sum over 32^3 cells.
"""
import numpy as np
import pytest
import torch

from tests.gpu_util import dev, ensure_lib

pytestmark = pytest.mark.gpu

N = 32


@pytest.fixture(scope="module")
def ctx():
    return ensure_lib().Context(N, 100.0, "fp64")


@pytest.mark.parametrize("lo,width,nbins", [
    (-6.0, 0.05, 240), (-3.0, 0.5, 1), (-8.0, 1.0 / 256, 4096), (0.1, 2.0 ** -30, 4000),
    (0.1, 2.0 ** -31, 4000), (-40.0, 0.7, 100), (31.5, 0.25, 7), (-1e3, 300.0, 9), (-6.0, 1e7, 3)])
def test_bins_and_moments(ctx, lo, width, nbins):
    rng = np.random.default_rng(nbins)
    x = rng.uniform(lo - 2 * min(width, 1.0), lo + (nbins + 2) * width, N ** 3).clip(-33, 33)
    x[: N ** 3 // 2] = 1.5 * rng.standard_normal(N ** 3 // 2)
    u = np.exp(x)
    edge = np.exp((lo + width * rng.integers(0, nbins + 1, 2000)).clip(-33, 33))
    u[:2000] = np.nextafter(edge, np.where(rng.random(2000) < 0.5, 0.0, np.inf))
    u[2000:4000] = edge
    u[4000:4200] = 1.0 + 2.0 ** rng.uniform(-52, -3, 200)
    u[4200:4206] = [1.0, 0.0, -0.5, 1e-200, 2.0 ** 60, 1.0 - 2.0 ** -53]
    delta = u - 1.0
    u = 1.0 + delta                          # as the library forms it
    counts, outside, moments = ctx.log_stats(dev(delta.reshape(N, N, N), torch.float64), lo, width,
                                             nbins)
    valid = u > 0
    ln = np.log(u[valid])
    t = (ln - lo) / width
    unsure = np.abs(t - np.rint(t)) * width <= 4 * np.spacing(np.maximum(np.abs(ln), abs(lo)))
    j = np.floor(t).clip(-1, nbins).astype(int)
    sure = np.bincount(j[~unsure] + 1, minlength=nbins + 2)
    either = np.zeros(nbins + 2, dtype=int)          # cells that may fall on either side
    for k in np.rint(t[unsure]).clip(-1, nbins + 1).astype(int):
        for b in {max(k - 1, -1), min(k, nbins)}:
            either[b + 1] += 1
    got = np.concatenate([[outside[0]], counts, [outside[1]]])
    assert outside[2] == int((~valid).sum())
    assert got.sum() + outside[2] == N ** 3
    assert np.all(got >= sure) and np.all(got <= sure + either)
    c = ln - ln.mean()
    var = (c * c).mean()
    want = [ln.mean(), var, (c ** 3).mean() / var ** 1.5, (c ** 4).mean() / var ** 2 - 3.0]
    np.testing.assert_allclose(moments, want, rtol=1e-12, atol=1e-12)
