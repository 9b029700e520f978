"""Which FP32 calls run the y and z passes of a plane in one kernel: the launches
of one Hessian-vector product, and, where a batch takes the plane kernel and a
solve by itself does not, the same bits from both.
"""
import pytest
import torch

from tests.gpu_util import dev, ensure_lib, pk_table_for, small_mock

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def plc():
    return ensure_lib()


@pytest.mark.parametrize("n,f1,f2,launches", [(72, 0, 0, 3), (96, 0, 0, 5), (96, 12, 8, 3), (108, 0, 0, 5),
                                              (128, 16, 8, 5), (128, 0, 0, 5)])
def test_launches_of_a_product(plc, n, f1, f2, launches):
    c = plc.Context(n, 6.0 * n, "mixed")
    k, P = pk_table_for(n, 6.0 * n)
    c.set_prior(k, P, -0.3)
    c.set_fft_schedule(f1, f2)
    x = torch.zeros((n, n, n), device="cuda")
    c.profile_enable(timing=False)
    c.hessvec(x, None, 1.0, x)
    assert sum(v[0] for v in c.profile_read().values()) == launches


def test_batch_of_108_gives_the_bits_of_single_solves(plc):
    ms = [small_mock(108, sigma=1.2, nbar=1.0, seed=s) for s in (1, 2)]
    cs = [plc.Context(m.n, m.box, "mixed") for m in ms]
    for c, m in zip(cs, ms):
        c.set_prior(m.k_tab, m.P_tab, m.mu)
    N = [dev(m.N, torch.int32) for m in ms]
    one = [c.newton_krylov_map(Ni, None, m.nbar).s for c, Ni, m in zip(cs, N, ms)]
    s = [torch.empty_like(o) for o in one]
    plc.Batch(cs).map(N, None, [m.nbar for m in ms], s, start=2)
    for got, want in zip(s, one):
        assert torch.equal(got, want)
