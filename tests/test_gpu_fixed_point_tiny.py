"""Values far below the quantum of the fixed-point FP64 passes: they count as
nothing, not as one quantum of a fixed sign (and fields of subnormals, which have
a quantum of their own, keep their value).

Bars.  The fields are chosen so that the passes are exact or round in one known
place; an error of one quantum in every element of a line then shows.
"""
import numpy as np
import pytest
import torch

from tests.gpu_util import ensure_lib, pk_table_for

pytestmark = pytest.mark.gpu

SIDES = [32, 64, 96, 128, 192, 256]


@pytest.fixture(scope="module")
def plc():
    return ensure_lib()


def _context(plc, n):
    c = plc.Context(n, 5.0 * n, "fp64")
    k, P = pk_table_for(n, 5.0 * n, seed=n)
    c.set_prior(k, P, -0.2)
    return c


# (the inverse of 192 = 16 x 12 takes this wave through a radix 3, which rounds)
@pytest.mark.parametrize("n", [n for n in SIDES if n != 192])
def test_zero_planes_add_nothing(plc, n):
    # (-1)^y on the plane z = 0, zero elsewhere: only the modes (0, n/2, kz)
    # are not zero, so the result is v(z) (-1)^y.  All-zero lines lie beside
    # the one that is not in the tiles of every pass.  Past the inverse y
    # transform, which gives +-v exactly, v and -v are shifted once (a tie
    # rounds up: they part by at most one quantum, which is below 2^-59 of the
    # largest v of the 16 planes that share an exponent; twice that allowed)
    # and rounded to double (half an ulp each).
    c = _context(plc, n)
    sign = 1.0 - 2.0 * (torch.arange(n, device="cuda", dtype=torch.float64) % 2)
    x = torch.zeros((n, n, n), dtype=torch.float64, device="cuda")
    x[0] = sign[:, None]
    y = c.prior_apply(x)
    v = y[:, 0, 0].abs()
    top = v.view(-1, 16).amax(1).repeat_interleave(16)
    off = (y - y[:, :1, :1] * sign[None, :, None]).abs().amax((1, 2))
    assert bool((v > 0).any())
    assert bool((off <= 2.0 ** -58 * top + 2.0 ** -52 * v).all())


@pytest.mark.parametrize("n", SIDES)
def test_vanishing_multipliers_add_nothing(plc, n):
    # a constant plus a wave of y at the highest frequency, smoothed by a
    # Gaussian that leaves nothing of the wave: a constant, to the last bit
    c = _context(plc, n)
    sign = 1.0 - 2.0 * (torch.arange(n, device="cuda", dtype=torch.float64) % 2)
    x = (1.5 + sign)[None, :, None].expand(n, n, n).contiguous()
    y = c.smooth(x, 5.0 * n)
    assert torch.equal(y, torch.full_like(y, float(y[0, 0, 0])))
    assert abs(float(y[0, 0, 0]) - 1.5) <= 1e-15


@pytest.mark.parametrize("n", SIDES)
def test_a_background_below_the_quantum_adds_nothing(plc, n):
    # 1e-300 beside 1 is nothing in double as in the passes: the same bits
    c = _context(plc, n)
    x = torch.zeros((n, n, n), dtype=torch.float64, device="cuda")
    x[n // 2, 1, n - 1] = 1.0
    y = c.prior_apply(x)
    for tiny in (1e-300, -1e-300, 1e-30):
        b = torch.where(x == 0.0, torch.full_like(x, tiny), x)
        assert torch.equal(c.prior_apply(b), y)


@pytest.mark.parametrize("n", SIDES)
def test_subnormal_fields(plc, n):
    # P(k) constant: y = 3.125 x.  All of x lies below 2^-1022, whose smallest
    # unit is 2^-1074; the passes' quantum follows the field down to 2^-1083, so
    # that their errors stay below a unit; the last rounding adds half a one.
    # Four allowed (x itself is 2^44 of them).
    c = plc.Context(n, 5.0 * n, "fp64")
    k, _ = pk_table_for(n, 5.0 * n)
    c.set_prior(k, np.full_like(k, 40.0), 0.0, 125.0 / 40.0)
    gen = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn((n, n, n), dtype=torch.float64, device="cuda", generator=gen) * 2.0 ** -1030
    assert 0.0 < float(x.abs().max()) < 2.0 ** -1022
    off = (c.prior_apply(x) * 2.0 ** 600 - 3.125 * (x * 2.0 ** 600)).abs().max()
    assert float(off) <= 4.0 * 2.0 ** (600 - 1074)
