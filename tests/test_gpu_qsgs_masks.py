"""QSGS growth by words of 32 cells against the host generator, byte for byte:
rows that end inside a word, one-cell rows, columns and planes (a cell is its
own neighbour there), targets reached in the seeding sweep, exactly, never,
and over more sweeps than the device runs between two looks of the host;
growing codes that stay allowed; a region; probabilities at the ends of
their range."""
import numpy as np
import pytest

from paper_1410_1914_gb300 import inputs

pytestmark = pytest.mark.gpu

SHAPES = [(5, 4, 1), (1, 1, 70), (3, 1, 2), (4, 7, 31), (4, 5, 32), (3, 4, 33), (1, 9, 64), (6, 1, 65), (9, 8, 100)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("case", [
    dict(code=1, allowed=[0], grown=[1], share=0.4, c_d=0.05, p=0.05),
    dict(code=1, allowed=[0], grown=[1], share=0.03, c_d=0.2, p=0.01),
    dict(code=2, allowed=[0, 3], grown=[1, 2], share=0.5, c_d=0.0, p=0.02),
    dict(code=1, allowed=[0], grown=[1], share=1.0, c_d=0.02, p=1.0),
    dict(code=1, allowed=[0], grown=[1], share=0.6, c_d=1.0, p=0.0),
    dict(code=3, allowed=[0, 1], grown=[3], share=0.9, c_d=0.1, p=0.0, sweeps=9),
    dict(code=1, allowed=[0, 2], grown=[1], share=0.5, c_d=0.05, p=0.1, sweeps=0)])
def test_growth_matches_host(cuda_lib, shape, case):
    import torch

    from paper_1410_1914_gb300 import _lib as L
    rng = np.random.default_rng(sum(shape) + case["code"])
    n = int(np.prod(shape))
    start = rng.choice(np.array([0, 0, 0, 0, 1, 2, 3], np.uint8), size=shape)
    region = (rng.random(shape) < 0.7).astype(np.uint8)
    bits = lambda codes: sum(1 << c for c in codes)
    for reg in (None, region):
        g, h = torch.from_numpy(start).cuda(), start.copy()
        target, sweeps = int(round(case["share"] * n)), case.get("sweeps", 60)
        args = (target, case["c_d"], case["p"], 17, 4)
        ng = L.cl_qsgs_grow(g, case["code"], bits(case["allowed"]), bits(case["grown"]), *args,
                            region=None if reg is None else torch.from_numpy(reg).cuda(), max_sweeps=sweeps)
        nh = inputs.grow(h, case["code"], case["allowed"], case["grown"], *args, region=reg, max_sweeps=sweeps)
        assert ng == nh
        np.testing.assert_array_equal(g.cpu().numpy(), h)


def test_growing_code_that_stays_allowed(cuda_lib):
    """A converted cell that may convert again counts again, as on the host."""
    import torch

    from paper_1410_1914_gb300 import _lib as L
    start = np.zeros((3, 4, 37), np.uint8)
    g, h = torch.from_numpy(start).cuda(), start.copy()
    assert L.cl_qsgs_grow(g, 1, 0b11, 0b10, 150, 0.1, 0.05, 3, 2, max_sweeps=40) == \
        inputs.grow(h, 1, [0, 1], [1], 150, 0.1, 0.05, 3, 2, max_sweeps=40)
    np.testing.assert_array_equal(g.cpu().numpy(), h)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("fraction", [0.0, 1e-300, 0.3, 1.0])
def test_faces_match_host(cuda_lib, shape, fraction):
    import torch

    from paper_1410_1914_gb300 import structures
    ph = np.random.default_rng(5).choice(np.array([0, 0, 1, 2], np.uint8), size=shape)
    np.testing.assert_array_equal(structures.reactive_faces(torch.from_numpy(ph).cuda(), fraction, 8).cpu().numpy(),
                                  inputs.reactive_faces(ph, fraction, 8))
