"""The FP32 kernels that run the y and z passes of a whole kx plane in one
block: register form (default schedules up to 96^3, and 128^3 inside a batch)
and Stockham form (other lengths up to 108^3), against the FP64 oracle at the
FP32 bars of the other operator tests (every element within 2e-5 of the
reference's largest, relative L2 within 1e-5).  They do the same operations on
the same values as the three passes, so a solve in a batch, which takes the
plane kernel at 128^3, gives the bits of a solve by itself, which does not.
"""
import numpy as np
import pytest
import torch

from oracle import plc as orc
from tests.gpu_util import dev, ensure_lib, host, max_rel, pk_table_for, rel_l2, small_mock

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def plc():
    return ensure_lib()


@pytest.mark.parametrize("n,f1,f2", [(4, 0, 0), (16, 0, 0), (32, 8, 4), (36, 0, 0), (64, 8, 8), (64, 0, 0),
                                     (72, 0, 0), (96, 8, 12), (96, 0, 0), (108, 0, 0), (144, 0, 0)])
def test_operator(plc, n, f1, f2):
    c = plc.Context(n, 6.0 * n, "mixed")
    k, P = pk_table_for(n, 6.0 * n, seed=n)
    c.set_prior(k, P, -0.3, 0.4)
    c.set_fft_schedule(f1, f2)
    x = np.random.default_rng(n).standard_normal((n, n, n))
    ref = orc.apply_Sinv(x, orc.inverse_eigenvalues(n, 6.0 * n, k, P, 0.4))
    y = host(c.prior_apply(dev(x, torch.float32)))
    assert rel_l2(y, ref) <= 1e-5 and max_rel(y, ref) <= 2e-5


def test_batch_of_128_gives_the_bits_of_single_solves(plc):
    ms = [small_mock(n, sigma=1.2, nbar=1.0, seed=n) for n in (128, 96, 128)]
    cs = [plc.Context(m.n, m.box, "mixed") for m in ms]
    for c, m in zip(cs, ms):
        c.set_prior(m.k_tab, m.P_tab, m.mu)
    N = [dev(m.N, torch.int32) for m in ms]
    one = [c.newton_krylov_map(Ni, None, m.nbar).s for c, Ni, m in zip(cs, N, ms)]
    s = [torch.empty_like(o) for o in one]
    b = plc.Batch(cs)
    b.map(N, None, [m.nbar for m in ms], s, start=2)
    for got, want in zip(s, one):
        assert torch.equal(got, want)
