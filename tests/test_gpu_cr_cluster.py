"""Cyclic-reduction slab solves on clusters: P and P^T against the oracle.

The sizes are the edges of the split: n_tot just above and below a power of
two (a level more or less), fewer block rows than a cluster of eight holds
comfortably, a single slab (no first pass), block rows that do not divide by
the cluster, 16- and 32-wide slabs, and groups of four right-hand sides that
are full, ragged and single.  FP64 to 1e-10 (the elimination orders differ by
rounding times condition numbers up to 1e4), mixed precision to 1e-4; a
right-hand side's result does not depend on its group: bit for bit.
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


# (n, b_pml, b_slab, fronts): n_tot = n + 2 + 2 b_pml
CASES = [(4, 2, 6, 1), (5, 2, 3, 1), (22, 4, 4, 2), (23, 4, 4, 1), (37, 12, 5, 2), (40, 12, 4, 1), (103, 12, 4, 2)]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,b_pml,b_slab,fronts", CASES)
def test_sweep_equals_oracle(n, b_pml, b_slab, fronts, precision):
    from paper_1705_09443_gb300 import LSSolver
    om = 2 * math.pi * (n + 1) / 8
    m = synth.gaussian_medium(n, 2, 4, 0.1, (0.8, 1.2), 11 + n)
    s = LSSolver(n, om, torch.tensor(m, dtype=torch.float64, device="cuda"), b_pml=b_pml, b_slab=b_slab,
                 precision=precision, fronts=fronts)
    pb = O.Problem2D(n, om, m, O.Params(b_pml=b_pml, b_slab=b_slab, fronts=fronts))
    rng = np.random.default_rng(n)
    R = 6
    x = rng.standard_normal((R, n, n)) + 1j * rng.standard_normal((R, n, n))
    xd = torch.tensor(x, dtype=torch.complex128, device="cuda")
    for tr in (False, True) if fronts == 1 else (False,):
        y = s.apply_P(xd, transpose=tr)
        for k in (1, 4, 5):   # the same columns in other groups
            assert torch.equal(s.apply_P(xd[:k], transpose=tr), y[:k]), (tr, k)
        y = y.cpu().numpy()
        for r in (0, 3, R - 1):
            ref = pb.precondition_transpose(x[r]) if tr else pb.precondition(x[r])
            assert rel(y[r], ref) <= (1e-4 if precision else 1e-10), (tr, r)
