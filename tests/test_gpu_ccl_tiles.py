"""Labelling by 32 x 8 x 8 tiles: boxes at and around the tile edges, dense and
sparse random phases, both neighbourhoods, with and without wrapping."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 8, 32), (9, 9, 33), (16, 16, 64), (7, 17, 65), (24, 8, 31), (2, 2, 96),
                                   (40, 33, 129)])
@pytest.mark.parametrize("nb,periodic", [(26, False), (26, True), (6, False), (6, True)])
def test_labels_and_statistics(cuda_lib, shape, nb, periodic):
    from paper_1410_1914_gb300 import _lib as L
    rng = np.random.default_rng(sum(shape) + nb + periodic)
    for share in (0.08, 0.3, 0.6):   # around the site-percolation thresholds of 26 and 6 neighbours, and above both
        ph = (rng.random(shape) < share).astype(np.uint8)
        lab = np.zeros(shape, np.int32)
        st = L.cl_phase_connectivity(ph, (1,), nb, periodic, lab)
        olab, ost = oracle.phase_connectivity(ph, (1,), nb, periodic)
        np.testing.assert_array_equal(lab, olab)
        assert st == ost
