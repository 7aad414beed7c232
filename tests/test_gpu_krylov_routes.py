"""The preconditioned Krylov solve over every route of its resident kernels:
the number of active cells selects a cluster or the whole grid, 2 to 8 cells
per thread in registers or vectors in memory (conjugate gradients), and 1 to 8
float4 per thread or memory (Gram-Schmidt)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,edge", [("d3q7", e) for e in (9, 33, 36, 70, 78, 86, 94, 100, 110, 116, 128)] +
                                         [("d3q19", e) for e in (9, 34, 72, 84, 96)])
def test_every_route_reaches_the_steady_state(cuda_lib, lattice, edge):
    from paper_1410_1914_gb300 import Solver, structures
    shape = (edge, edge + 1, edge - 1)   # ragged rows and planes
    ph = structures.pt_cl(shape, 3 + edge, 0.45, 0.188743)
    params = dict(dx_m=2e-9, knudsen=1, T_K=353.0, bc_in=0, bc_out=0, c_in=1.0, c_out=0.0, check_every=200)
    s = Solver(shape, storage="fp32pop", lattice=lattice, **params)
    s.set_structure(ph)
    a = s.solve_krylov_dsa(tol=1e-8, max_iter=2000, max_steps=0)
    assert 0 < a["iterations"] <= 600
    f = s.fluxes()
    C = s.field()
    # at the steady state what enters leaves, through every plane, to the rounding of f32 populations
    assert f["J_in"] > 0 and abs(f["J_in"] - f["J_out"]) < 1e-4 * f["J_in"]
    # the solve repeats bit by bit (fixed-order sums)
    s.init()
    b = s.solve_krylov_dsa(tol=1e-8, max_iter=2000, max_steps=0)
    assert (a["iterations"], a["inner_iterations"]) == (b["iterations"], b["inner_iterations"])
    np.testing.assert_array_equal(C, s.field())
    # and is where the time march stays: 200 steps change nothing beyond f32 rounding of C <= 1
    s.step(200)
    assert float(np.abs(s.field() - C).max()) < 200 * 6e-8 * 4
    s.close()
