"""The host's twiddle table of the fixed-point FP64 passes (no GPU): entries
against cos and sin in 50 digits, and none for lengths without those passes.

An entry is the nearest integer to w 2^61 of a long double with an error of at
most 2^-63 in w (64 significant bits): off by at most 0.5 + 0.25.
"""
import subprocess
from decimal import Decimal, localcontext

import pytest

from paper_0911_1407_gb300 import build

MAIN = r"""
#include <cstdio>
#include "passesx.cuh"
int main() {
  for (int n = 4; n <= 512; n += 2) {
    const auto tw = plc::fx_twiddles(n);
    std::printf("n %d %d\n", n, (int)tw.size());
    auto val = [](plc::fxk k) { return ((long long)k.h << 32) + k.l; };
    for (const plc::fxw& w : tw) std::printf("%lld %lld %lld\n", val(w.c), val(w.m), val(w.p));
  }
}
"""


def _cos_sin(m, n):
    """cos and sin of 2 pi m / n by their series, argument below pi / 4."""
    pi = Decimal("3.14159265358979323846264338327950288419716939937510")
    octant, r = divmod(8 * m, n)
    odd = octant & 1
    x = 2 * pi * (n - r if odd else r) / (8 * n)
    c = s = Decimal(0)
    t = Decimal(1)
    for k in range(40):
        if k % 2 == 0:
            c += t * (1 - k % 4)
        else:
            s += t * (2 - k % 4)
        t = t * x / (k + 1)
    c, s = (s, c) if odd else (c, s)
    for _ in range(octant // 2):      # quarter turns
        c, s = -s, c
    return c, s


@pytest.fixture(autouse=True)
def _fifty_digits():
    with localcontext() as c:
        c.prec = 50
        yield


def test_the_series():
    for m, n, c, s in ((0, 32, 1, 0), (8, 32, 0, 1), (16, 32, -1, 0), (24, 32, 0, -1)):
        a, b = _cos_sin(m, n)
        assert abs(a - c) < Decimal("1e-38") and abs(b - s) < Decimal("1e-38")
    a, b = _cos_sin(5, 12)      # 150 degrees
    assert abs(b - Decimal("0.5")) < Decimal("1e-38") and a < 0 and abs(4 * a * a - 3) < Decimal("1e-37")


def test_twiddles(tmp_path):
    src, exe = tmp_path / "tw.cu", tmp_path / "tw"
    src.write_text(MAIN)
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, str(src), "-o",
                    str(exe)], check=True, capture_output=True, timeout=600)
    out = iter(subprocess.run([str(exe)], check=True, capture_output=True, text=True,
                              timeout=60).stdout.splitlines())
    for line in out:
        _, n, size = line.split()
        n, size = int(n), int(size)
        assert size == (n if n in (32, 64, 96, 128, 192, 256) else 0)
        for m in range(size):
            c, dm, dp = map(int, next(out).split())
            d = dm + c
            assert dp == c + d
            ec, es = _cos_sin(m, n)
            assert abs(c - ec * 2 ** 61) <= Decimal("0.75"), (n, m)
            assert abs(d + es * 2 ** 61) <= Decimal("0.75"), (n, m)
