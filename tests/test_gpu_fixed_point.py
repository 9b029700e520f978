"""The FP64 passes in 64-bit block fixed point (lengths with a four-step
schedule) against the FP64 Stockham passes of the same context.

Bars.  Both forms round each of the five passes at about 2^-53 of a line's
norm; the fixed-point tiles at 2^-54 or below, so where the result is known
their relative L2 error may not exceed the Stockham form's by more than the
scatter of one such sum (a tenth).  The two forms agree to the sum
of both errors, at most 60 roundings of 2^-53 of the result's norm in L2 for
fields whose transform does not cancel (7e-15).  Scaling by a power of two
moves every tile's exponent and changes no integer, so it is exact.
"""
import numpy as np
import pytest
import torch

from tests.gpu_util import dev, ensure_lib, host, pk_table_for

pytestmark = pytest.mark.gpu

DEFAULT = {32: (8, 4), 64: (8, 8), 96: (12, 8), 128: (16, 8), 192: (16, 12), 256: (16, 16)}


@pytest.fixture(scope="module")
def plc():
    return ensure_lib()


def _context(plc, n):
    c = plc.Context(n, 5.0 * n, "fp64")
    k, P = pk_table_for(n, 5.0 * n, seed=n)
    c.set_prior(k, P, -0.2)
    return c


def _fields(n, rng):
    x = rng.standard_normal((n, n, n))
    impulse = np.zeros((n, n, n))
    impulse[1, n - 1, n // 2] = 1.0
    slab = np.zeros((n, n, n))
    slab[n - 1] = x[0]                      # most tiles all zero
    return {"noise": x, "spiky": np.exp(3.0 * x), "impulse": impulse, "slab": slab,
            "uneven": x * np.exp(12.0 * rng.standard_normal((n, 1, 1)))}


@pytest.mark.parametrize("n", [32, 64, 128])
def test_no_less_accurate_than_fp64_passes(plc, n):
    # P(k) constant and the DC mode at the same eigenvalue: S^-1 is c times
    # the identity (c known to rounding only, so fitted), and what is left of
    # y - c x is the rounding of the passes
    c = plc.Context(n, 5.0 * n, "fp64")
    k, _ = pk_table_for(n, 5.0 * n)
    c.set_prior(k, np.full_like(k, 40.0), 0.0, 125.0 / 40.0)
    for name, x in _fields(n, np.random.default_rng(n)).items():
        xl, err = x.astype(np.longdouble), {}
        for f in (DEFAULT[n], (0, 0)):
            c.set_fft_schedule(*f)
            y = host(c.prior_apply(dev(x, torch.float64))).astype(np.longdouble)
            d = y - (xl * y).sum() / (xl * xl).sum() * xl
            err[f] = float(np.sqrt((d * d).sum() / (y * y).sum()))
        assert err[DEFAULT[n]] <= 1.1 * err[(0, 0)], (name, err)


@pytest.mark.parametrize("n", sorted(DEFAULT))
def test_matches_the_stockham_passes(plc, n):
    c = _context(plc, n)
    rng = np.random.default_rng(n)
    x = torch.from_numpy(rng.standard_normal((n, n, n))).cuda()
    s = -0.2 + 0.5 * x
    N = torch.from_numpy(rng.poisson(1.0, (n, n, n)).astype(np.int32)).cuda()
    got = {}
    for f in (DEFAULT[n], (0, 0)):
        c.set_fft_schedule(*f)
        y = x.clone()
        c.prior_apply(y, y)                 # in place
        f_val, g = c.logpost_grad(s, N, None, 1.3)
        got[f] = [y, c.hessvec(s, None, 1.3, x), g, torch.tensor(f_val, dtype=torch.float64)]
    for a, b in zip(got[DEFAULT[n]], got[(0, 0)]):
        assert float((a - b).norm()) <= 7e-15 * float(b.norm())


def test_scaling_by_a_power_of_two_is_exact(plc):
    c = _context(plc, 64)
    x = torch.from_numpy(np.exp(2.0 * np.random.default_rng(5).standard_normal((64, 64, 64)))).cuda()
    y = c.prior_apply(x)
    for p in (-700, -60, 60, 700):
        assert torch.equal(c.prior_apply(x * 2.0 ** p), y * 2.0 ** p)


@pytest.mark.parametrize("n", [32, 96])
def test_zero_and_non_finite_fields(plc, n):
    c = _context(plc, n)
    x = torch.zeros((n, n, n), dtype=torch.float64, device="cuda")
    assert torch.equal(c.prior_apply(x), x)
    for bad in (float("nan"), float("inf"), -float("inf")):
        x.normal_()
        x[n - 1, 0, n - 1] = bad
        assert not bool(torch.isfinite(c.prior_apply(x)).any())
    x.normal_()
    assert bool(torch.isfinite(c.prior_apply(x)).all())   # nothing of it stays behind


def test_exponential_to_the_last_place(plc):
    # a constant v lies in the DC mode, whose eigenvalue is infinite, so
    # H v = nbar e^s v exactly.  Within |s| < 32 the integer exponential is one
    # rounding (half an ulp) of a value within 2^-56.6 (0.09 ulp); outside the
    # library function allows one ulp.
    n = 32
    c = _context(plc, n)
    rng = np.random.default_rng(3)
    s = np.concatenate([rng.uniform(-33, 33, n ** 3 // 2), 3.0 * rng.standard_normal(n ** 3 // 2)])
    edge = [0.0, -0.0, 1e-300, -5e-324, 2.0 ** -60, -2.0 ** -53, 31.999999999999996, -31.999999999999996,
            32.0, -32.0, 40.0, 709.7, 710.0, -700.0, -746.0, np.log(2.0), np.log(2.0) / 128,
            -np.log(2.0) / 128, float("inf"), -float("inf"), float("nan")]
    s[:len(edge)] = edge
    one = torch.ones((n, n, n), dtype=torch.float64, device="cuda")
    y = host(c.hessvec(dev(s.reshape(n, n, n), torch.float64), None, 1.0, one)).ravel()
    with np.errstate(over="ignore", under="ignore"):
        ref = np.exp(s.astype(np.longdouble))
        want = ref.astype(np.float64)
    assert np.array_equal(np.isnan(y), np.isnan(want))
    inf = np.isinf(want)
    assert np.array_equal(y[inf], want[inf])
    ok = np.isfinite(want)
    ulps = np.abs(y[ok].astype(np.longdouble) - ref[ok]) / np.spacing(want[ok])
    assert float(np.max(ulps[np.abs(s[ok]) < 32])) <= 0.6
    assert float(np.max(ulps)) <= 1.0
