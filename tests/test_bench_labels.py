"""The bench names the slab solver that a leg runs."""
import pytest


@pytest.mark.parametrize("dim,R,prec,label", [(2, 64, 1, "block LU"), (2, 16, 1, "block LU"), (2, 15, 1, "block cyclic"),
                                              (2, 64, 0, "block cyclic"), (2, 16, 0, "block cyclic"),
                                              (3, 16, 1, "block elimination")])
def test_slab_solver_label(dim, R, prec, label):
    import bench
    assert bench.slab_solver(dim, R, prec).startswith(label)
