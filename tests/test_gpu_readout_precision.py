"""Per-plane readouts as good as sums in FP64.

After an initialisation with the linear field the state is known exactly (C is
the ramp of the half-way faces, as a pair of floats or one float; the
deviations are zero), so the mean of a plane is that value and its consumption
the number of its catalytic links times w C (1 - r), whatever the number of
cells.  A plane of a box with `rows` rows is added up in FP64 over at most
ceil(rows / 64) shares of eight warps: 8 + rows / 64 additions, the flush of a
share, and a few products, each off by at most u = 2^-53."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,lattice", [(s, l) for l in ("d3q7", "d3q19") for s in ("fp32", "fp16dev", "fp32pop")])
@pytest.mark.parametrize("shape", [(5, 24, 96), (40, 50, 33)])
def test_plane_sums_against_the_known_state(cuda_lib, storage, lattice, shape):
    from paper_1410_1914_gb300 import Solver
    nz, ny, nx = shape
    rng = np.random.default_rng(3)
    ph = (rng.random(shape) < 0.2).astype(np.uint8)   # isolated solid cells in an open box
    c_in, c_out = 0.9371, 0.2113
    s = Solver(shape, storage=storage, lattice=lattice, dx_m=2e-9, D_bulk=2e-5, knudsen=0, T_K=353.0, bc_in=0, bc_out=0,
               c_in=c_in, c_out=c_out, k_ms=1e3, react_rule=1, check_every=20)
    s.set_structure(ph)
    total, R, C = s.reaction_rate()
    info = s.info()
    _, reactive = s.links()
    s.close()
    x = np.arange(nx)
    if storage != "fp32pop" and lattice == "d3q7":   # the plane march takes f32 boundary values
        ci, co = float(np.float32(c_in)), float(np.float32(c_out))
    else:
        ci, co = c_in, c_out
    ramp = ci + (co - ci) * (x + 0.5) / nx
    hi = ramp.astype(np.float32)
    q = 7 if lattice == "d3q7" else 19
    w = np.array([1 / 8] * 6 if q == 7 else [1 / 18] * 6 + [1 / 36] * 12, np.float32)
    w0 = np.float32(1 / 4 if q == 7 else 1 / 3)
    nlinks = np.stack([((reactive >> i) & 1).sum(axis=(0, 1)) for i in range(q - 1)]).astype(np.float64)  # [q - 1][nx]
    if storage == "fp32pop":   # populations w C, rounded
        g = np.concatenate([[w0], w])[:, None] * hi[None, :]
        if q == 7:   # C is the f32 sum of the populations, in the step's order
            v = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + g[6])
            Cx = v.astype(np.float64)
        else:
            Cx = g.astype(np.float64).sum(axis=0)
        part = (nlinks * g[1:].astype(np.float64)).sum(axis=0)
    else:
        lo = (ramp - hi.astype(np.float64)).astype(np.float32)
        if storage == "fp16dev" and q == 7:   # scaled by 2^(38 - E), c < 2^E
            lo = (lo.astype(np.float64) * 2.0 ** 38).astype(np.float16).astype(np.float64) * 2.0 ** -38
        Cx = hi.astype(np.float64) + lo
        part = (nlinks * w[:, None].astype(np.float64)).sum(axis=0) * Cx
    rows = ny * nz
    adds = 8 + (rows + 63) // 64 + 4
    u = 2.0 ** -53
    np.testing.assert_allclose(C, Cx, rtol=adds * u, atol=0)
    cs2 = 0.25 if q == 7 else 1 / 3
    sink = 2.0 * info["k_lu"] / (cs2 + info["k_lu"])
    exp = part * sink * (2e-9 ** 3 / info["dt_s"])
    np.testing.assert_allclose(R, exp, rtol=(adds + 8) * u, atol=0)
