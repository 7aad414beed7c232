"""Calls that take a cluster of 16 blocks, where no such cluster can be placed
(CL_LBM_NO_CLUSTER=1 takes that way on any device): the steady solves of small
systems on the grid must reach what the cluster's route reaches, and the bias
gradient is summed by one block per channel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _solve(kind, edge, lattice):
    from paper_1410_1914_gb300 import Solver, structures
    shape = (edge, edge + 1, edge - 1)
    s = Solver(shape, storage="fp32pop", lattice=lattice, dx_m=2e-9, knudsen=1, T_K=353.0, bc_in=0, bc_out=0, c_in=1.0,
               c_out=0.0, check_every=20)
    s.set_structure(structures.pt_cl(shape, 5, 0.45, 0.188743))
    if kind == "lines":
        info = s.solve_steady_lines(tol=1e-10, max_iter=500, restart=200, cg_tol=1e-3)
        assert info["status"] == "CL_OK"
    else:
        info = s.solve_krylov_dsa(tol=1e-8, max_iter=1000, max_steps=0)
    out = info["iterations"], info["inner_iterations"], s.field()
    s.close()
    return out


# 6: one block; 12: a few blocks of one cell per thread; 25: two cells per thread in a full cluster
@pytest.mark.parametrize("kind,lattice", [("dsa", "d3q7"), ("dsa", "d3q19"), ("lines", "d3q7")])
@pytest.mark.parametrize("edge", [6, 12, 25])
def test_small_systems_on_the_grid(cuda_lib, monkeypatch, kind, lattice, edge):
    a = _solve(kind, edge, lattice)
    monkeypatch.setenv("CL_LBM_NO_CLUSTER", "1")
    b = _solve(kind, edge, lattice)
    if kind == "dsa":   # the same blocks, the same order of sums
        assert a[:2] == b[:2]
        np.testing.assert_array_equal(a[2], b[2])
    else:               # residuals of 1e-10: fields to the rounding of f32
        assert abs(a[0] - b[0]) <= 2
        np.testing.assert_allclose(a[2], b[2], rtol=0, atol=4 * 6e-8)


def test_bias_gradient_without_a_cluster(cuda_lib, monkeypatch):
    import torch

    from paper_1410_1914_gb300 import warmstart as W
    gen = torch.Generator(device="cuda").manual_seed(3)
    dy = torch.randint(-3, 4, (20000, 24), device="cuda", generator=gen).to(torch.bfloat16)
    db = torch.full((16,), 7.0, device="cuda")
    monkeypatch.setenv("CL_LBM_NO_CLUSTER", "1")
    W._call("cl_nn_bias_grad", W._p(dy), 20000, 16, 24, 8, W._p(db), None)
    torch.cuda.synchronize()
    assert torch.equal(db.double(), dy[:, 8:].double().sum(0))   # whole numbers below 2^24: exact in any order
