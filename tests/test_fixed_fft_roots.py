"""The roots of unity of the fixed-point transforms, from their first octant.

Against 40-digit arithmetic, for every line length, as the integers that the
digits are made from (units of 2^-62): within one unit (half from rounding to
integers, a quarter each at most from the function and its angle below pi / 4 on
a 64-bit mantissa).  The axes are exact.
"""
import decimal
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
SRC = r"""
#include <cstdio>
#include <vector>
#include "fx_line.cuh"
int main() {
    for (int lg = kFxMinLg; lg <= kFxMaxLg; ++lg) {
        const int L = 1 << lg;
        std::vector<long double> c(L), s(L);
        fx_host_roots(L, c.data(), s.data());
        for (int k = 0; k < L; ++k)
            printf("%d %d %lld %lld\n", L, k, (long long)llrintl(ldexpl(c[k], 62)), (long long)llrintl(ldexpl(s[k], 62)));
    }
    return 0;
}
"""


def exact(L):
    """exp(-2 pi i k / L), k < L, by repeated multiplication in 40 digits."""
    D = decimal.Decimal
    re, im = D(-1), D(0)                      # exp(-i pi), halved down to exp(-2 pi i / L)
    for _ in range(L.bit_length() - 2):
        re, im = ((1 + re) / 2).sqrt(), -((1 - re) / 2).sqrt()
    out = [(D(1), D(0))]
    for _ in range(L - 1):
        a, b = out[-1]
        out.append((a * re - b * im, a * im + b * re))
    return out


def test_roots_of_unity(tmp_path):
    if not os.path.exists(NVCC):
        pytest.skip("no nvcc")
    (tmp_path / "roots.cu").write_text(SRC)
    exe = str(tmp_path / "roots")
    subprocess.run([NVCC, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I",
                    os.path.join(ROOT, "paper_1705_09443_gb300", "csrc"), str(tmp_path / "roots.cu"), "-o", exe],
                   check=True)
    got = {}
    for line in subprocess.run([exe], capture_output=True, text=True, check=True).stdout.splitlines():
        L, k, c, s = map(int, line.split())
        got.setdefault(L, []).append((c, s))
    assert sorted(got) == [64, 128, 256, 512, 1024, 2048]
    with decimal.localcontext() as ctx:
        ctx.prec = 40
        for L, roots in got.items():
            assert len(roots) == L
            for k, (g, e) in enumerate(zip(roots, exact(L))):
                for a, b in zip(g, e):
                    assert abs(a - b * 2 ** 62) <= 1, (L, k)
            q, one = L // 4, 2 ** 62
            assert roots[0] == (one, 0) and roots[q] == (0, -one) and roots[2 * q] == (-one, 0) and roots[3 * q] == (0, one)
