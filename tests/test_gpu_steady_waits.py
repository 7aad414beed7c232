"""Bounded waits of the steady solves (gpu), made to run out on purpose.

The resident kernels of the two preconditioned solves meet as a whole grid; a
block waits for the others for a limited time.  The hook shortens the limit
and makes a meeting one that never comes about, or one that a single block
misses while all others make it: the last meeting of a Gram-Schmidt, after
which the other blocks finish as if nothing had happened.  Either way the call
returns CL_ERR_TIMEOUT, the state is what it was, and the handle solves as a
fresh one once the hook is reset.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHORT = 100_000  # SM clock cycles


def _solver(lattice, edge):
    from paper_1410_1914_gb300 import Solver, structures
    shape = (edge, edge + 1, edge - 1)
    s = Solver(shape, storage="fp32pop", lattice=lattice, dx_m=2e-9, knudsen=1, T_K=353.0, bc_in=0, bc_out=0,
               c_in=1.0, c_out=0.0, check_every=20)
    s.set_structure(structures.pt_cl(shape, 5, 0.45, 0.188743))
    return s


def _solve(s, solver):
    if solver == "lines":
        return s.solve_steady_lines(tol=1e-8, max_iter=20, restart=20, cg_tol=1e-3)
    return s.solve_krylov_dsa(tol=1e-8, max_iter=20, max_steps=0)


# 40^3: the conjugate gradients of either solve take the whole grid; 16^3: only the Gram-Schmidt does
@pytest.mark.parametrize("solver,lattice,edge,never", [("dsa", "d3q7", 40, 1), ("dsa", "d3q7", 40, 2),
                                                       ("dsa", "d3q7", 16, 1), ("dsa", "d3q7", 16, 2),
                                                       ("dsa", "d3q19", 40, 1), ("dsa", "d3q19", 40, 2),
                                                       ("lines", "d3q7", 40, 1)])
def test_a_wait_that_runs_out_is_reported(cuda_lib, solver, lattice, edge, never):
    from paper_1410_1914_gb300 import _lib as L
    lib = L.load()
    s = _solver(lattice, edge)
    before = s.populations()
    assert lib.cl_lbm_set_wait_test(s.h, SHORT, never) == L.CL_OK
    with pytest.raises(L.ClError) as e:
        _solve(s, solver)
    assert e.value.status == L.CL_ERR_TIMEOUT
    np.testing.assert_array_equal(s.populations(), before)
    assert lib.cl_lbm_set_wait_test(s.h, 0, 0) == L.CL_OK
    a = _solve(s, solver)
    ref = _solver(lattice, edge)
    b = _solve(ref, solver)
    assert a["iterations"] == b["iterations"] > 0
    np.testing.assert_array_equal(s.populations(), ref.populations())
    s.close()
    ref.close()
