"""The LS operator's fixed-point FFT passes at the edges of their line lengths.

The reference is the oracle's FFT convolution in complex128.  Both sides carry
a few 1e-16 of transform error and the kernel weights agree to about 1e-14
relative (their arguments reach several hundred), so 1e-13 in the relative
2-norm bounds the difference with room for neither a wrong entry nor a lost
low digit.
"""
import math

import numpy as np
import pytest

from oracle import lss_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-13


def _solver(n, dim=2, seed=0):
    from paper_1705_09443_gb300 import LSSolver, LSS_MIXED
    rng = np.random.default_rng(seed)
    m = 0.3 * rng.uniform(-1, 1, (n,) * dim)
    om = 2 * math.pi * n / (8 if dim == 2 else 4)
    s = LSSolver(n, om, torch.tensor(m, device="cuda"), b_pml=4, b_slab=4, precision=LSS_MIXED, factor=False)
    return s, m, om


def _field(n, dim, R, seed=1):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((R,) + (n,) * dim) + 1j * rng.standard_normal((R,) + (n,) * dim)


def _err(y, ref):
    return float(np.linalg.norm(y - ref) / np.linalg.norm(ref))


# n = 17 .. 1024: first and last size of each line length 64 .. 2048, four and
# eight entries per thread, odd numbers of right-hand sides
@pytest.mark.parametrize("n,R", [(17, 1), (32, 3), (33, 1), (64, 1), (64, 41), (65, 2), (128, 5), (129, 1), (256, 1),
                                 (256, 2), (257, 1), (511, 3), (512, 1), (513, 1), (1024, 1)])
@pytest.mark.parametrize("transpose", [False, True])
def test_operator_2d(n, R, transpose):
    if transpose and n > 300:
        pytest.skip("the transpose differs in the first and last pass only")
    s, m, om = _solver(n)
    kw = O.nystrom_weights(2, n, om, n)
    x = _field(n, 2, R)
    y = s.apply_A(torch.tensor(x, device="cuda"), transpose=transpose).cpu().numpy()
    for r in {0, R - 1}:
        ref = (O.ls_apply_transpose if transpose else O.ls_apply)(x[r], m, om, kw)
        assert _err(y[r], ref) < TOL


@pytest.mark.parametrize("n,R", [(17, 1), (24, 3), (33, 2), (65, 1)])
def test_operator_3d(n, R):
    s, m, om = _solver(n, 3)
    kw = O.nystrom_weights(3, n, om, n)
    x = _field(n, 3, R)
    y = s.apply_A(torch.tensor(x, device="cuda")).cpu().numpy()
    ref = O.ls_apply(x[R - 1], m, om, kw)
    assert _err(y[R - 1], ref) < TOL


@pytest.mark.parametrize("kind", ["spike", "checkerboard", "rows", "zero"])
def test_uneven_fields(kind):
    """One entry, the highest frequency, rows that differ by 1e12, nothing."""
    n = 100
    s, m, om = _solver(n)
    x = np.zeros((1, n, n), dtype=np.complex128)
    if kind == "spike":
        x[0, 37, 91] = 0.7 - 0.2j
    elif kind == "checkerboard":
        x[0] = (-1.0) ** np.add.outer(np.arange(n), np.arange(n))
    elif kind == "rows":
        x = _field(n, 2, 1) * np.logspace(0, -12, n)[None, :, None]
    y = s.apply_A(torch.tensor(x, device="cuda")).cpu().numpy()
    if kind == "zero":
        assert not y.any()
        return
    assert _err(y[0], O.ls_apply(x[0], m, om, O.nystrom_weights(2, n, om, n))) < TOL


@pytest.mark.parametrize("n,dim", [(40, 2), (150, 2), (20, 3)])
def test_power_of_two_scaling_is_exact(n, dim):
    """The arithmetic is scale-free: 2^k x gives 2^k y bit for bit."""
    s, _, _ = _solver(n, dim)
    x = torch.tensor(_field(n, dim, 2), device="cuda")
    y = s.apply_A(x)
    for k in (-900, 900):
        assert torch.equal(s.apply_A(x * 2.0 ** k), y * 2.0 ** k)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("n,dim", [(64, 2), (20, 3)])
def test_non_finite_input(n, dim, bad):
    """A non-finite entry makes its own right-hand side non-finite and no other."""
    s, _, _ = _solver(n, dim)
    x = torch.tensor(_field(n, dim, 3), device="cuda")
    y0 = s.apply_A(x)
    x[(1,) + (5,) * dim] = bad
    y = s.apply_A(x)
    assert not torch.isfinite(torch.view_as_real(y[1])).any()
    assert torch.equal(y[0], y0[0]) and torch.equal(y[2], y0[2])


@pytest.mark.parametrize("n,dim", [(40, 2), (300, 2), (20, 3)])
def test_plane_wave_rhs(n, dim):
    s, m, om = _solver(n, dim)
    rng = np.random.default_rng(3)
    d = rng.standard_normal((3, dim))
    d /= np.linalg.norm(d, axis=1)[:, None]
    g, uI = s.plane_wave_rhs(d, with_incident=True)
    kw = O.nystrom_weights(dim, n, om, n)
    tol = TOL + 4 * np.finfo(float).eps * om * math.sqrt(dim)   # rounding of the phase on both sides
    assert _err(uI[2].cpu().numpy(), O.plane_wave(n, om, d[2])) < tol
    assert _err(g[2].cpu().numpy(), O.ls_rhs(m, om, kw, d[2])) < tol
