"""Cluster slab solves where every slab is wider than 16 layers.

The cluster's size and threads follow the number of clusters of a pass (slabs
times groups of right-hand sides).  With four slabs (three of 24 layers), in FP64: 8 CTAs up to 4
right-hand sides, 4 from 5 to 9, two CTAs per SM from 10, clusters of 2 from 77.
The same columns have to come out bit for bit in all of them, and as the oracle
has them (FP64 to 1e-10, mixed to 1e-4).  20 and 24 layers: the columns beyond
are left out in FP64.
"""
import math

import numpy as np
import pytest

from oracle import lss_oracle as O
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,b_pml,b_slab", [(30, 12, 8), (30, 12, 12)])
def test_every_cluster_size(n, b_pml, b_slab, precision):
    from paper_1705_09443_gb300 import LSSolver
    om = 2 * math.pi * (n + 1) / 8
    m = synth.gaussian_medium(n, 2, 4, 0.1, (0.8, 1.2), n)
    s = LSSolver(n, om, torch.tensor(m, device="cuda"), b_pml=b_pml, b_slab=b_slab, precision=precision)
    widths = [s.slab_info(i)[1] + s.slab_info(i)[2] for i in range(s.n_slabs)]
    assert min(widths) > 16
    pb = O.Problem2D(n, om, m, O.Params(b_pml=b_pml, b_slab=b_slab))
    rng = np.random.default_rng(n)
    x = rng.standard_normal((100, n, n)) + 1j * rng.standard_normal((100, n, n))
    xd = torch.tensor(x, device="cuda")
    for tr in (False, True):
        y = s.apply_P(xd, transpose=tr)
        for R in (1, 4, 5, 9, 10, 16, 17, 40, 76, 77):
            assert torch.equal(s.apply_P(xd[:R], transpose=tr), y[:R]), (tr, R)
        for r in (0, 99):
            ref = pb.precondition_transpose(x[r]) if tr else pb.precondition(x[r])
            assert np.linalg.norm(y[r].cpu().numpy() - ref) <= (1e-4 if precision else 1e-10) * np.linalg.norm(ref)
