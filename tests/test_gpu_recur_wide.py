"""Interface recurrences of many right-hand sides against those of few.

Every right-hand side is independent, so P on R of them must equal P on four
at a time, which the cluster chains or the row form of the recurrences serve.
The slab solves are held to the cyclic reduction, so only the recurrences'
order of summation differs: sums of n_tot products, a few hundred roundings at
most over the slabs, 1e-12 in FP64 and 1e-5 in single precision.
"""
import math

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(n, R, fronts, precision, b_pml, transpose=False):
    from paper_1705_09443_gb300 import LSSolver
    m = synth.gaussian_medium(n, 2, 4, 0.08, (0.8, 1.2), 1706)
    s = LSSolver(n, 2 * math.pi * n / 8, torch.tensor(m, device="cuda"), b_pml=b_pml, b_slab=4, precision=precision,
                 fronts=fronts)
    rng = np.random.default_rng(5)
    x = torch.tensor(rng.standard_normal((R, n, n)) + 1j * rng.standard_normal((R, n, n)), device="cuda")
    y = s.apply_P(x, transpose=transpose)
    rows = sorted({0, R // 2, R - 1})
    for r in rows:
        lo = min(r, R - 4)
        ref = s.apply_P(x[lo:lo + 4].contiguous(), transpose=transpose)[r - lo]
        err = float(torch.linalg.vector_norm(y[r] - ref) / torch.linalg.vector_norm(ref))
        assert err < (1e-12 if precision == 0 else 1e-5), (r, err)


# 16-, 32- and 64-column tiles, full and ragged, one and several of them
@pytest.mark.parametrize("R", [9, 16, 17, 33, 65])
@pytest.mark.parametrize("fronts", [1, 2])
def test_column_tiles_fp64(R, fronts, monkeypatch):
    monkeypatch.setenv("LSS_SLAB_SOLVE", "cr")
    _check(256, R, fronts, 0, 12)


@pytest.mark.parametrize("R,fronts", [(24, 1), (40, 2), (97, 2)])
def test_column_tiles_mixed(R, fronts, monkeypatch):
    monkeypatch.setenv("LSS_SLAB_SOLVE", "cr")
    _check(301, R, fronts, 1, 12)


# two and three slabs (the middle slab first, or with one neighbour on each side), one row per task
@pytest.mark.parametrize("n,R", [(6, 401), (10, 301), (24, 301)])
@pytest.mark.parametrize("fronts", [1, 2])
@pytest.mark.parametrize("precision", [0, 1])
def test_few_slabs(n, R, fronts, precision, monkeypatch):
    monkeypatch.setenv("LSS_SLAB_SOLVE", "cr")
    _check(n, R if precision == 0 else 2 * R, fronts, precision, 4)


def test_transposed_sweep(monkeypatch):
    monkeypatch.setenv("LSS_SLAB_SOLVE", "cr")
    _check(200, 21, 1, 0, 12, transpose=True)
