"""The FP32 four-step passes of the largest grid (512 = 32 x 16: two rounds of
paired x-pass tasks and of phase-B tasks per block) against the FP64 operators
on the same inputs, and the Stockham schedule beside them.  Bars as for the
other FP32 operators: every element within 2e-5 of the reference's largest,
relative L2 within 1e-5.
"""
import pytest
import torch

from tests.gpu_util import ensure_lib, pk_table_for

pytestmark = pytest.mark.gpu


def _close(a, ref):
    d = a.double() - ref
    return float(d.norm()) <= 1e-5 * float(ref.norm()) and \
        float(d.abs().max()) <= 2e-5 * float(ref.abs().max())


def test_operators_at_512():
    plc = ensure_lib()
    n = 512
    k, P = pk_table_for(n, 5.0 * n)
    gen = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((n, n, n), device="cuda", generator=gen)
    s = -0.3 + 0.5 * torch.randn((n, n, n), device="cuda", generator=gen)
    w = torch.rand((n, n, n), device="cuda", generator=gen)
    with plc.Context(n, 5.0 * n, "fp64") as c:
        c.set_prior(k, P, -0.3)
        ref_y = c.prior_apply(x.double())
        ref_h = c.hessvec(s.double(), w.double(), 1.2, x.double())
    with plc.Context(n, 5.0 * n, "mixed") as c:
        c.set_prior(k, P, -0.3)
        for f in ((32, 16), (0, 0)):
            c.set_fft_schedule(*f)
            assert _close(c.prior_apply(x), ref_y), f
            assert _close(c.hessvec(s, w, 1.2, x), ref_h), f
