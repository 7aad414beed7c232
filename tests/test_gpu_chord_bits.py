"""Pore lengths from bit masks against the oracle's: rows of one word and of
several with ragged ends, boxes whose loops close after one and after many
turns, open boxes and slabs (runs of the whole box, crossed 16 cells at a
time), and rows too short for the masks (the line kernels)."""
import numpy as np
import pytest

import oracle
from paper_1410_1914_gb300 import inputs

pytestmark = pytest.mark.gpu

SHAPES = [(9, 7, 14), (8, 8, 31), (8, 8, 32), (12, 10, 33), (33, 17, 65), (7, 64, 96), (40, 1, 40), (1, 36, 50),
          (16, 16, 13), (24, 36, 130)]


def _compare(ph, **extra):
    from paper_1410_1914_gb300 import Solver
    params = dict(dx_m=2e-9, knudsen=1, T_K=353.0, bc_in=0, bc_out=0, c_in=1.0, c_out=0.0, k_ms=0.0, **extra)
    s = Solver(ph.shape, **params)
    s.set_structure(ph)
    o = oracle.OracleLBM(ph, **params)
    i = s.info()
    pores = (ph == 0) | (ph == 3)
    assert i["mean_pore_diameter_m"] == pytest.approx(oracle.pore_diameter(ph, params["dx_m"])[pores].mean(), rel=1e-12)
    assert i["D_max"] == pytest.approx(o.D_max, rel=1e-12)
    om = s.setup()["omega"]
    act = o.active() > 0
    np.testing.assert_array_equal(om > 0, act)
    # omega is the f32 rounding of the FP64 value: half an ulp, and one where the FP64 values round apart
    np.testing.assert_allclose(om[act], 1.0 / o.tau()[act], rtol=1.2e-7, atol=0)
    s.close()


@pytest.mark.parametrize("shape", SHAPES)
def test_layers(cuda_lib, shape):
    ph = inputs.pt_cl(shape, 5 + sum(shape), 0.5, 0.2, c_d=0.02)
    ph[:, :, 0] = 0
    _compare(ph)


@pytest.mark.parametrize("shape", SHAPES)
def test_open_boxes_and_slabs(cuda_lib, shape):
    ph = np.zeros(shape, np.uint8)
    _compare(ph)                                # every loop closed, every run the box
    ph[shape[0] // 2, :, 1:] = 1                # one solid plane but for the inlet
    _compare(ph)
    ph = np.zeros(shape, np.uint8)
    ph[:, :, shape[2] // 2:] = 2                # pores and transporting ionomer
    _compare(ph, D_ionomer=1e-9)
