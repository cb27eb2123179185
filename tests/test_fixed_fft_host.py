"""Error of the fixed-point line transforms, compiled for the host, against
transforms in long double (tests/fixed_fft_host.cu).

A line's convolution with a kernel line that passes a resonance, as in the
operator's column pass, for every line length and both plans.
 - noise: no entry is worse than the others.  An entry's error is a sum of many
   roundings with mean zero, so the root mean square of 64 lines' errors at one
   index is within 9 % (one sigma) of that over all indexes; a rounding with a
   mean adds up at index 0 (6 to 9 times).  Bound: 1.6, more than six sigma.
 - noise, and a line of alternating sign, whose transform is largest where the
   kernel is smallest: the error is no larger than that of double transforms.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
LINES = 64


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("no nvcc")
    exe = str(tmp_path_factory.mktemp("fx") / "fixed_fft_host")
    subprocess.run([NVCC, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I",
                    os.path.join(ROOT, "paper_1705_09443_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "fixed_fft_host.cu"), "-o", exe], check=True)
    return exe


def rms(a):
    return float(np.sqrt((np.abs(a) ** 2).mean()))


def errors(exe, lg, entries, x):
    L = 1 << lg
    j = np.minimum(np.arange(L), L - np.arange(L))
    kernel = (1.0 / (1.0 - (j / (L / 8 + 0.3)) ** 2) / L).astype(np.complex128)
    data = np.ascontiguousarray(x, dtype=np.complex128).tobytes() + kernel.tobytes()
    out = subprocess.run([exe, str(lg), str(entries), str(LINES)], input=data, capture_output=True, check=True).stdout
    q = np.frombuffer(out, dtype=np.complex128).reshape(LINES, 3, L // 2)
    return q[:, 0], q[:, 1]


@pytest.mark.parametrize("lg,entries", [(6, 4), (7, 8), (8, 8), (9, 8), (10, 4), (10, 8), (11, 8)])
def test_error_of_a_line_convolution(harness, lg, entries):
    n = 1 << (lg - 1)
    rng = np.random.default_rng(lg)
    fixed, double = errors(harness, lg, entries, rng.standard_normal((LINES, n)) + 1j * rng.standard_normal((LINES, n)))
    assert rms(fixed[:, 0]) <= 1.6 * rms(fixed)
    assert rms(fixed) <= rms(double)
    phase = np.exp(2j * np.pi * rng.random((LINES, 1)))
    fixed, double = errors(harness, lg, entries, phase * (-1.0) ** np.arange(n))
    assert rms(fixed) <= rms(double)
