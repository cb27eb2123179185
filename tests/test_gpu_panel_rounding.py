"""Rounding of the 3D pivot panels: how far the mixed-precision P is from FP64.

The difference is the rounding of the FP32 pivot-block inversions.  Mean over
twelve media at n = 9: 3.72e-7 with every entry's update rounded once at its own
size (as the factorization did before the panels went to registers), 4.11e-7
rounded twice, each mean known to 0.04e-7.  Bound between them: 3.92e-7.
"""
import math

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_mixed_factors_round_once_per_update(monkeypatch):
    from paper_1705_09443_gb300 import LSSolver
    monkeypatch.setenv("LSS_TC_UPDATE", "0")
    n, err = 9, []
    for seed in range(12):
        m = torch.tensor(synth.gaussian_medium(n, 3, 4, 0.15, (0.8, 1.2), 50 + seed), device="cuda")
        g = torch.Generator("cuda").manual_seed(seed)
        x = torch.randn((2, n, n, n), dtype=torch.complex128, device="cuda", generator=g)
        y = [LSSolver(n, 2 * math.pi * n / 4, m, b_pml=4, precision=p).apply_P(x) for p in (0, 1)]
        err.append(float(torch.linalg.norm((y[1] - y[0]).flatten()) / torch.linalg.norm(y[0].flatten())))
    assert np.mean(err) <= 3.92e-7, err
