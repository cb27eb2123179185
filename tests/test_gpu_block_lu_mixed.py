"""Block LU slab solves where they are used: mixed precision, R >= 16.

The 16-wide slabs go to the block LU, the 32-wide ones to the cyclic reduction
on clusters beside it (LSS_SLAB_SOLVE=cr sends every slab there).  Partial
column groups (R = 17, 20, 33), full ones, one and two fronts, ragged last
slabs and the fronts meeting in slab 0.  Both are FP32 eliminations of the same
subproblems in another order: within 1e-5 of each other and 1e-4 of the oracle,
and not bit for bit the same, which shows that the block LU ran.
"""
import math

import numpy as np
import pytest

from oracle import lss_oracle as O
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def make(n, b_pml, b_slab, fronts, seed):
    from paper_1705_09443_gb300 import LSS_MIXED, LSSolver
    om = 2 * math.pi * (n + 1) / 8
    m = synth.gaussian_medium(n, 2, 4, 0.1, (0.8, 1.2), seed)
    s = LSSolver(n, om, torch.tensor(m, dtype=torch.float64, device="cuda"), b_pml=b_pml, b_slab=b_slab,
                 precision=LSS_MIXED, fronts=fronts)
    return s, m, om


@pytest.mark.parametrize("n,b_pml,b_slab,fronts,R", [(64, 12, 4, 2, 16), (64, 12, 4, 1, 20), (50, 8, 3, 2, 33),
                                                     (37, 6, 4, 1, 64), (9, 3, 3, 2, 16), (100, 12, 5, 2, 17)])
def test_block_lu_equals_cyclic_reduction_mixed(n, b_pml, b_slab, fronts, R, monkeypatch):
    s, m, om = make(n, b_pml, b_slab, fronts, 3 + n)
    rng = np.random.default_rng(5 + R)
    x = rng.standard_normal((R, n, n)) + 1j * rng.standard_normal((R, n, n))
    xd = torch.tensor(x, dtype=torch.complex128, device="cuda")
    monkeypatch.setenv("LSS_SLAB_SOLVE", "cr")
    y_cr = s.apply_P(xd).cpu().numpy()
    monkeypatch.delenv("LSS_SLAB_SOLVE")
    y_lu = s.apply_P(xd).cpu().numpy()
    assert not np.array_equal(y_lu, y_cr)
    pb = O.Problem2D(n, om, m, O.Params(b_pml=b_pml, b_slab=b_slab, fronts=fronts))
    for r in range(R):
        assert rel(y_lu[r], y_cr[r]) <= 1e-5, r
    for r in (0, R - 1):
        assert rel(y_lu[r], pb.precondition(x[r])) <= 1e-4, r


def test_wide_slab_runs_beside_the_block_lu():
    """The middle slab's clusters must not wait for the block LU of the others:
    pass A with twice the right-hand sides (neither fills the GPU alone) took
    twice the time when they did, 1.1 times it beside them."""
    s, _, _ = make(128, 12, 4, 2, 7)
    ms = []
    for R in (32, 64):
        x = torch.randn((R, 128, 128), dtype=torch.complex128, device="cuda")
        s.apply_P(x)
        t = []
        for _ in range(9):
            s.profile_read()
            s.profile(True)
            s.apply_P(x)
            t.append(s.profile_read()[0]["slab_a"])
            s.profile(False)
        ms.append(sorted(t)[4])
    assert ms[1] <= 1.5 * ms[0], ms
