"""The bounded wait of the 3D tensor-core update when it expires for some warps
of a CTA and not for others: the CTA leaves as a whole, the call returns the
timeout status and the context goes on working.

The waits are only reported as expired (the products themselves have
completed), so nothing is left in flight.
"""
import math

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# M = (b_slab + b_pml) n_tot: one tile per slab, and several with a ragged last one
@pytest.mark.parametrize("n", [6, 20])
def test_partly_expired_wait_ends_with_timeout(n):
    from paper_1705_09443_gb300 import GmresOptions, LSS_MIXED, LssError, LSSolver
    m = synth.gaussian_medium(n, 3, 3, 0.15, (0.8, 1.2), 63)
    s = LSSolver(n, 2 * math.pi * (n + 1) / 8, torch.tensor(m, dtype=torch.float64, device="cuda"), b_pml=3, b_slab=3,
                 precision=LSS_MIXED)
    g = s.plane_wave_rhs(np.eye(3)[:1])
    u0, _ = s.solve(g, GmresOptions(30, 1e-8, 100))
    with pytest.raises(LssError) as e:
        s.test_inject(3)
    assert e.value.code == -6
    u1, st = s.solve(g, GmresOptions(30, 1e-8, 100))   # the factors were not touched
    assert st[0]["converged"] and torch.equal(u0, u1)


def test_other_contexts_are_refused():
    from paper_1705_09443_gb300 import LssError, LSSolver
    s = LSSolver(16, 13.0, torch.zeros((16, 16), dtype=torch.float64, device="cuda"), b_pml=4, b_slab=4, factor=False)
    with pytest.raises(LssError) as e:
        s.test_inject(3)
    assert e.value.code == -1
