"""omega = 1 / tau is rounded to f32 from a value as good as FP64: where 1 / tau
lies 16 u (u = 2^-53) from the middle between two floats, it goes to the nearer
one.  tau = 1/2 + D / (2 D_max) is exact for these D (D_max = 1, tau_ref = 1)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,lattice", [("fp32", "d3q7"), ("fp32pop", "d3q19")])
def test_relaxation_rates_next_to_ties(cuda_lib, storage, lattice):
    from paper_1410_1914_gb300 import Solver
    rng = np.random.default_rng(4)
    shape = (16, 17, 18)
    n = int(np.prod(shape))
    f = (1 + rng.random(n) * 0.99).astype(np.float32)                 # omega in (1, 2)
    up = np.nextafter(f, np.float32(3))
    mid = (f.astype(np.float64) + up.astype(np.float64)) / 2
    side = rng.integers(0, 2, n)
    tau = (1 / mid) * np.where(side, 1 - 16 * 2.0 ** -53, 1 + 16 * 2.0 ** -53)   # 1 / tau above or below the middle
    D = 2 * tau - 1
    assert (0.5 + 0.5 * D == tau).all() and (D > 0).all() and (D < 1).all()
    D[0] = 1.0
    s = Solver(shape, storage=storage, lattice=lattice, dx_m=2e-9, D_bulk=2e-5, knudsen=0, bc_in=0, bc_out=0, tau_ref=1.0,
               check_every=20)
    s.set_structure(np.zeros(shape, np.uint8))
    s.set_diffusivity(D.reshape(shape))
    om = s.setup()["omega"].ravel()
    s.close()
    np.testing.assert_array_equal(om[1:], np.where(side, up, f)[1:])
