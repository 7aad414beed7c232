"""J_in, J_out and R of the reducing step as good as sums in FP64: with the FP32
state they are sums of the very values that the readout of that state adds up.
Each side adds exact terms, at most 40 additions in FP64 deep (the threads of a
block, the blocks, the shares of rows, the planes), and the readout's boundary
terms take four FP64 roundings each; u = 2^-53."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice", ["d3q7", "d3q19"])
@pytest.mark.parametrize("shape", [(300, 9, 64), (96, 40, 70), (64, 64, 64)])
def test_fluxes_of_the_reducing_step_equal_the_readout(cuda_lib, lattice, shape):
    from paper_1410_1914_gb300 import Solver
    nz, ny, nx = shape
    ph = (np.random.default_rng(nx).random(shape) < 0.25).astype(np.uint8)
    ph[..., 0] = 0
    s = Solver(shape, storage="fp32", lattice=lattice, dx_m=1e-8, D_bulk=1e-5, k_ms=400.0, react_rule=1, c_in=0.7371,
               c_out=0.1113, bc_in=0, bc_out=0, check_every=20)
    s.set_structure(ph)
    before = s.field().astype(np.float64)
    info = s.solve_budget(20)
    f = s.fluxes()
    after = s.field().astype(np.float64)
    s.close()
    u = 2.0 ** -53
    w = 2 / 8 if lattice == "d3q7" else 2 * (1 / 18 + 4 / 36)   # of the links through a face, twice
    faces = ny * nz * w * 2 * 0.7371                            # sum of the terms' magnitudes
    assert abs(info["J_in"] - f["J_in"]) <= (80 + 8) * u * faces
    assert abs(info["J_out"] - f["J_out"]) <= (80 + 8) * u * faces
    assert f["R"] > 0 and abs(info["R"] - f["R"]) <= 80 * u * f["R"]
    if lattice == "d3q19":   # the residual's sums too (the plane march adds those in f32 per thread)
        resid = np.abs(after - before).sum() / np.abs(after).sum()
        assert abs(info["resid"] - resid) <= 2 * 80 * u * resid
