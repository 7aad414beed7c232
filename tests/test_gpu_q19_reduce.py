"""The reducing D3Q19 step's sums (kept in pairs of floats down to the warp)
against the readout of the state it leaves, FP32 state.  Both sum the same
FP32 values of C = hi + lo and of the deviations; a pair carries at least 40
bits, so a sum of n terms of size t differs by at most n t 2^-40.  Rows of
32 and 64 cells per warp, pairs that straddle the end of an odd row, boundary
values that FP32 does not hold exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 2), (5, 6, 33), (3, 9, 64), (4, 7, 97), (2, 17, 128), (3, 4, 161)])
@pytest.mark.parametrize("bc_out", [0, 1])
def test_reducing_step_equals_readout(cuda_lib, shape, bc_out):
    from paper_1410_1914_gb300 import Solver
    rng = np.random.default_rng(sum(shape))
    nz, ny, nx = shape
    ph = (rng.random(shape) < 0.25).astype(np.uint8)
    ph[..., 0] = 0
    react = rng.integers(0, 64, shape).astype(np.uint8)
    s = Solver(shape, storage="fp32", lattice="d3q19", dx_m=1e-8, D_bulk=1e-5, k_ms=40.0, c_in=0.7, c_out=0.1,
               bc_out=bc_out, check_every=6)
    s.set_structure(ph, react)
    s.init()
    info = s.solve_budget(6)
    f = s.fluxes()
    faces = 5 * ny * nz * 2.0 * 0.7 / 18.0 * 2.0 ** -40
    assert abs(info["J_in"] - f["J_in"]) <= faces
    assert abs(info["J_out"] - f["J_out"]) <= faces
    assert abs(info["R"] - f["R"]) <= 18 * nx * ny * nz * 0.7 / 18.0 * 2.0 ** -40
    s.close()
