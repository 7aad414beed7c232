"""The line-eliminated solve over every route of its resident conjugate
gradients (one cluster, the grid with 1 to 8 cells per thread, vectors in
memory), selected by the number of active cells."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 5), (3, 4, 6), (16, 15, 17), (20, 21, 22), (40, 41, 42), (50, 51, 49), (60, 61, 62),
                                   (72, 71, 70), (90, 91, 92)])
def test_every_route_reaches_the_linear_profile_of_an_open_box(cuda_lib, shape):
    # every cell a pore: F's fixed point is the linear profile between the half-way faces, D_eff = D_b
    from paper_1410_1914_gb300 import Solver
    nz, ny, nx = shape
    s = Solver(shape, storage="fp32pop", dx_m=2e-9, D_bulk=2e-5, knudsen=0, bc_in=0, bc_out=0, c_in=1.0, c_out=0.0)
    s.set_structure(np.zeros(shape, np.uint8))
    s.init(np.full(shape, 0.25, np.float32))   # not the answer
    info = s.solve_steady_lines(tol=1e-12, max_iter=200, restart=100, cg_tol=1e-3)
    assert info["status"] == "CL_OK", info
    x = 1.0 - (np.arange(nx) + 0.5) / nx
    np.testing.assert_allclose(s.field(), np.broadcast_to(x, shape), rtol=0, atol=4 * 6e-8)
    assert s.effective_diffusivity()[1] == pytest.approx(1.0, rel=1e-5)
    # FP64 fluxes of the result: J = D_b-flux through ny nz cells, cs^2 (tau - 1/2) = 1/8 per unit gradient 1/nx
    assert info["J_in"] == pytest.approx(ny * nz / (8.0 * nx), rel=1e-9)
    assert info["J_out"] == pytest.approx(info["J_in"], rel=1e-9)
    s.close()
