"""Populations of the D3Q19 (C, delta) state are w C + delta rounded to f32 once.
A uniform state C (delta = 0) with w C next to the middle between two floats
shows a second rounding: C = m / w in FP64 puts w C within 2^-48 of such a middle
m, and the exact side follows from whole numbers."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _to_f32(v):
    """The float nearest the fraction v > 0 (ties to even)."""
    e = 0
    while v >= 2:
        v, e = v / 2, e + 1
    while v < 1:
        v, e = v * 2, e - 1
    k = v * 2 ** 23
    n = k.numerator // k.denominator
    rest = k - n
    if rest > Fraction(1, 2) or (rest == Fraction(1, 2) and n & 1):
        n += 1
    return np.float32(np.ldexp(float(n), e - 23))


@pytest.mark.parametrize("storage", ["fp32", "fp16dev"])
def test_uniform_state_next_to_ties(cuda_lib, storage):
    from paper_1410_1914_gb300 import Solver
    rng = np.random.default_rng(9)
    weights = [np.float32(1 / 3)] + [np.float32(1 / 18)] * 6 + [np.float32(1 / 36)] * 12
    for w in (weights[0], weights[1], weights[7]):
        for _ in range(20):
            f = np.float32(0.02 + 0.01 * rng.random())
            mid = (float(f) + float(np.nextafter(f, np.float32(1)))) / 2      # exact in FP64
            C = mid / float(w)
            hi = np.float32(C)
            lo = np.float32(C - float(hi))
            s = Solver((2, 2, 3), storage=storage, lattice="d3q19", dx_m=2e-9, D_bulk=2e-5, knudsen=0, bc_in=0, bc_out=0,
                       c_in=C, c_out=C, check_every=20)
            s.set_structure(np.zeros((2, 2, 3), np.uint8))
            g = s.populations()
            s.close()
            exact = Fraction(float(hi)) + Fraction(float(lo))
            for i in (0, 1, 7):
                want = _to_f32(Fraction(float(weights[i])) * exact)
                assert (g[i] == want).all(), (float(w), i, g[i].ravel()[:3], want)
