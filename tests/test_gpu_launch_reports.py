"""What lss_autotune reports is what the launches use."""
import math

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def make(n, precision):
    from paper_1705_09443_gb300 import LSSolver
    m = synth.gaussian_medium(n, 2, 4, 0.08, (0.8, 1.2), 3)
    return LSSolver(n, 2 * math.pi * n / 8, torch.tensor(m, dtype=torch.float64, device="cuda"), b_pml=6,
                    precision=precision)


@pytest.mark.parametrize("precision,auto", [(0, 1), (1, 4)])
def test_right_hand_sides_per_cluster(precision, auto, monkeypatch):
    """LSS_SOLVE_NR=2 is read when the context is made; one right-hand side
    needs no group."""
    monkeypatch.delenv("LSS_SOLVE_NR", raising=False)
    s = make(24, precision)
    monkeypatch.setenv("LSS_SOLVE_NR", "2")
    t = make(24, precision)
    assert s.autotune(5)["solve_rhs_per_cta"] == auto and t.autotune(5)["solve_rhs_per_cta"] == 2
    assert s.autotune(1)["solve_rhs_per_cta"] == t.autotune(1)["solve_rhs_per_cta"] == 1
    x = torch.randn((5, 24, 24), dtype=torch.complex128, device="cuda")
    assert torch.equal(s.apply_P(x), t.apply_P(x))


@pytest.mark.parametrize("n,lines", [(17, 4), (100, 4), (256, 4), (257, 2), (700, 2)])
def test_lines_per_cta_of_the_operator(n, lines):
    """Padded lengths up to 512 have four lines per CTA, above two."""
    assert make(n, 1).autotune(1)["fft_col_group"] == lines
