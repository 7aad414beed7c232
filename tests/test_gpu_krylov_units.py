"""The preconditioned Krylov solve in any unit of concentration: the equation is
linear, so boundary values scaled by a power of two give the same iterates
scaled by it, bit for bit, as long as nothing leaves the range of f32."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice", ["d3q7", "d3q19"])
def test_steady_state_scales_with_the_boundary_values(cuda_lib, lattice):
    from paper_1410_1914_gb300 import Solver, structures
    shape = (20, 21, 22)
    ph = structures.pt_cl(shape, 8, 0.45, 0.188743)
    out = {}
    for e in (0, -60, 60, 90):   # 2^90 = 1.2e27, below the 1e30 that a handle takes
        s = Solver(shape, storage="fp32pop", lattice=lattice, dx_m=2e-9, knudsen=1, T_K=353.0, bc_in=0, bc_out=0,
                   c_in=2.0 ** e, c_out=2.0 ** (e - 2), k_ms=1e3, react_rule=1, check_every=20)
        s.set_structure(ph)
        info = s.solve_krylov_dsa(tol=1e-8, max_iter=1000, max_steps=0)
        f = s.fluxes()
        out[e] = (info["iterations"], info["inner_iterations"], np.ldexp(s.field().astype(np.float64), -e),
                  [np.ldexp(f[k], -e) for k in ("J_in", "J_out", "R")], s.effective_diffusivity()[1])
        s.close()
    for e in (-60, 60, 90):
        assert out[e][:2] == out[0][:2]
        np.testing.assert_array_equal(out[e][2], out[0][2])
        assert out[e][3:] == out[0][3:]
