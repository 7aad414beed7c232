"""The steady solves of small systems where no cluster of their size can be
placed: CL_LBM_NO_CLUSTER=1 takes the grid's route at every size, which must
reach what the cluster's reaches."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _solve(kind, edge, lattice):
    from paper_1410_1914_gb300 import Solver, structures
    shape = (edge, edge + 1, edge - 1)
    s = Solver(shape, storage="fp32pop", lattice=lattice, dx_m=2e-9, knudsen=1, T_K=353.0, bc_in=0, bc_out=0, c_in=1.0,
               c_out=0.0, check_every=20)
    s.set_structure(structures.pt_cl(shape, 5, 0.45, 0.188743))
    if kind == "lines":
        info = s.solve_steady_lines(tol=1e-10, max_iter=500, restart=200, cg_tol=1e-3)
        assert info["status"] == "CL_OK"
    else:
        info = s.solve_krylov_dsa(tol=1e-8, max_iter=1000, max_steps=0)
    out = info["iterations"], info["inner_iterations"], s.field()
    s.close()
    return out


# 6: one block; 12: a few blocks of one cell per thread; 25: two cells per thread in a full cluster
@pytest.mark.parametrize("kind,lattice", [("dsa", "d3q7"), ("dsa", "d3q19"), ("lines", "d3q7")])
@pytest.mark.parametrize("edge", [6, 12, 25])
def test_small_systems_on_the_grid(cuda_lib, monkeypatch, kind, lattice, edge):
    a = _solve(kind, edge, lattice)
    monkeypatch.setenv("CL_LBM_NO_CLUSTER", "1")
    b = _solve(kind, edge, lattice)
    if kind == "dsa":   # the same blocks, the same order of sums
        assert a[:2] == b[:2]
        np.testing.assert_array_equal(a[2], b[2])
    else:               # residuals of 1e-10: fields to the rounding of f32
        assert abs(a[0] - b[0]) <= 2
        np.testing.assert_allclose(a[2], b[2], rtol=0, atol=4 * 6e-8)
