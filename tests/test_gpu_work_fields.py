"""Device memory of a context's solver work: thirteen fields of n^3 doubles in
either precision (the FP64 CG's diagonal has no field of its own), taken by the
first call that needs any; and FP64 solves that use the shared one give the
bits of a context that has done nothing else.
"""
import pytest
import torch

from tests.gpu_util import dev, ensure_lib, small_mock

pytestmark = pytest.mark.gpu


def _taken(plc, precision, n):
    c = plc.Context(n, 5.0 * n, precision)
    x = torch.zeros((n, n, n), dtype=torch.float64, device="cuda")
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    c.smooth(x, 1.0, y)
    taken = before - torch.cuda.mem_get_info()[0]
    c.close()
    return taken


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_thirteen_fields(precision):
    plc, n = ensure_lib(), 128
    _taken(plc, precision, n)               # loads the kernels
    assert 12.5 * 8 * n ** 3 < _taken(plc, precision, n) < 13.5 * 8 * n ** 3


@pytest.mark.parametrize("n", [32, 48])
def test_fp64_solves_after_others(n):
    plc, m = ensure_lib(), small_mock(n, "radial_masked", sigma=1.0, nbar=2.0)
    N, w = dev(m.N, torch.int32), dev(m.w, torch.float64)
    u = torch.ones((n, n, n), dtype=torch.float64, device="cuda")

    def context():
        c = plc.Context(n, m.box, "fp64")
        c.set_prior(m.k_tab, m.P_tab, m.mu)
        return c
    calls = [lambda c: c.newton_krylov_map(N, w, m.nbar, tol=1e-8).s,
             lambda c: c.newton_krylov_map(N, w, m.nbar, tol=1e-8, device_driven=0).s,
             lambda c: c.wiener_lsq(N, w, m.nbar, tol=1e-8)[0],
             lambda c: c.gauss_map(N, w, m.nbar, tol=1e-6).s,
             lambda c: c.map_vjp(torch.zeros_like(u), w, m.nbar, u, tol=1e-8)[0],
             lambda c: c.smooth(u, 1.0)]
    alone = [call(context()) for call in calls]
    one = context()
    for _ in range(2):
        for call, want in zip(calls, alone):
            assert torch.equal(call(one), want)
