"""Routes that only large or elongated boxes take: the D3Q19 Laplacian's conjugate
gradients with five and eight cells per thread and with their vectors in memory,
and the convolution by gathers (more than 65535 planes in the batch)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("edge", [92, 110, 118])
def test_d3q19_krylov_with_many_cells_per_thread(cuda_lib, edge):
    from paper_1410_1914_gb300 import Solver, structures
    shape = (edge, edge + 1, edge - 1)   # ragged rows and planes
    s = Solver(shape, storage="fp32pop", lattice="d3q19", dx_m=2e-9, knudsen=1, T_K=353.0, bc_in=0, bc_out=0, c_in=1.0,
               c_out=0.0, check_every=200)
    s.set_structure(structures.pt_cl(shape, 3 + edge, 0.45, 0.188743))
    a = s.solve_krylov_dsa(tol=1e-8, max_iter=2000, max_steps=0)
    assert 0 < a["iterations"] <= 600
    f = s.fluxes()
    C = s.field()
    # what enters leaves, to the rounding of f32 populations; the march stays there (200 steps of f32 roundings of C <= 1)
    assert f["J_in"] > 0 and abs(f["J_in"] - f["J_out"]) < 1e-4 * f["J_in"]
    s.step(200)
    assert float(np.abs(s.field() - C).max()) < 200 * 6e-8 * 4
    s.close()


@pytest.mark.parametrize("ci,co,shape,periodic", [(16, 16, (1, 65537, 1, 2), 1), (80, 48, (3, 21846, 2, 1), 0)])
def test_forward_convolution_of_many_planes_exact(cuda_lib, ci, co, shape, periodic):
    # whole numbers: every sum is exact in f32, the result is rounded once to bf16
    import torch

    from paper_1410_1914_gb300 import warmstart as W
    gen = torch.Generator(device="cuda").manual_seed(ci)
    N, D, H, X = shape
    x = torch.randint(-2, 3, (N, D, H, X, ci), generator=gen, device="cuda").to(torch.bfloat16)
    w = torch.randint(-2, 3, (27, co, ci), generator=gen, device="cuda").to(torch.bfloat16)
    b = torch.randint(-9, 10, (co,), generator=gen, device="cuda").float()
    y = torch.empty(N, D, H, X, co, dtype=torch.bfloat16, device="cuda")
    W._call("cl_nn_conv3d", W._p(x), W._p(w), W._p(b), W._p(y), N, D, H, X, ci, co, ci, 0, co, 0, 1, periodic, None)
    W._call("cl_nn_check", None)
    ref = b.expand(N, D, H, X, co).clone()
    for t in range(27):
        v = x.float()
        for dim, d in ((3, t % 3 - 1), (2, t // 3 % 3 - 1), (1, t // 9 - 1)):
            if d == 0:
                continue
            v = torch.roll(v, -d, dim)
            if dim == 3 or not periodic:
                idx = [slice(None)] * 5
                idx[dim] = slice(-1, None) if d > 0 else slice(0, 1)
                v[tuple(idx)] = 0
        ref += v @ w[t].float().T
    assert torch.equal(y, ref.clamp(min=0).to(torch.bfloat16))
