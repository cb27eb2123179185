"""The operator's arithmetic is symmetric in the sign of the field, as FP64's is:
A(-x) = -A(x) and A^T(-x) = -A^T(x) bit for bit, since every rounding is to
nearest with ties to even.  A rounding with a direction (ties up, bits dropped)
shifts every entry the same way, which the sum of the two shows.
Sizes: one per line length, both plans, 2D and 3D.  Noise fields: a line's scale
may depend on the sign where its largest entry is an exact power of two.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dim,R", [(30, 2, 1), (64, 2, 1), (64, 2, 64), (100, 2, 2), (200, 2, 1), (259, 2, 1),
                                     (512, 2, 2), (700, 2, 1), (20, 3, 2), (64, 3, 1)])
def test_operator_is_odd(n, dim, R):
    from paper_1705_09443_gb300 import LSSolver
    rng = np.random.default_rng(n)
    m = torch.tensor(0.3 * rng.uniform(-1, 1, (n,) * dim), device="cuda")
    s = LSSolver(n, 2 * math.pi * n / (8 if dim == 2 else 4), m, b_pml=4, b_slab=4, factor=False)
    x = rng.standard_normal((R,) + (n,) * dim) + 1j * rng.standard_normal((R,) + (n,) * dim)
    x = torch.tensor(x, dtype=torch.complex128, device="cuda")
    for tr in (False, True):
        assert torch.equal(s.apply_A(-x, transpose=tr), -s.apply_A(x, transpose=tr))
