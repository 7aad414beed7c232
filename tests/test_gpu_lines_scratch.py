"""Device memory of a line-eliminated solve: what the header says, so that a box
that fits by it is not refused."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

USED_MEM_HIGH = 8   # cudaMemPoolAttrUsedMemHigh


def _cudart():
    for name in ("libcudart.so.13", "/usr/local/cuda/lib64/libcudart.so"):
        try:
            return ctypes.CDLL(name)
        except OSError:
            pass
    pytest.skip("no CUDA runtime library to ask")


@pytest.mark.parametrize("open_box", [True, False])
@pytest.mark.parametrize("restart", [3, 10])
def test_scratch_is_what_the_header_says(cuda_lib, open_box, restart):
    from paper_1410_1914_gb300 import Solver, structures
    rt = _cudart()
    pool = ctypes.c_void_p()
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    shape = (60, 61, 62)
    ph = np.zeros(shape, np.uint8) if open_box else structures.pt_cl(shape, 5, 0.45, 0.188743).cpu().numpy()
    s = Solver(shape, storage="fp32pop", dx_m=2e-9, knudsen=1, T_K=353.0, bc_in=0, bc_out=0, c_in=1.0, c_out=0.0)
    s.set_structure(ph)
    n, N = s.fluxes()["n_active"], ph.size
    # runs: active cells whose - neighbour is not one (or the face of the box), and loops of y and z
    act = s.setup()["active"].astype(bool)
    runs = sum(int((act & ~np.roll(act, 1, ax)).sum()) for ax in range(3)) + int(act[:, :, 0].sum())
    runs += int(act[:, 0].sum()) + int(act[0].sum())
    held, zero, high = ctypes.c_uint64(), ctypes.c_uint64(0), ctypes.c_uint64()
    assert rt.cudaMemPoolGetAttribute(pool, USED_MEM_HIGH - 1, ctypes.byref(held)) == 0
    assert rt.cudaMemPoolSetAttribute(pool, USED_MEM_HIGH, ctypes.byref(zero)) == 0
    s.solve_steady_lines(tol=1e-30, max_iter=restart, restart=restart, cg_tol=1e-1)
    assert rt.cudaMemPoolGetAttribute(pool, USED_MEM_HIGH, ctypes.byref(high)) == 0
    s.close()
    said = 8 * ((2 * restart + 28) * n + 7 * runs + N // 2 + 5 * n * (restart < 4))
    assert 0 < high.value - held.value <= said + (1 << 20)
