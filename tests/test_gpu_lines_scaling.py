"""The line-eliminated solve's cost per cell and iteration does not grow with the
box: every block of the Gram-Schmidt once added up the parts of all others,
which made an iteration of 160^3 cost 3.6 times as much per cell as one of 64^3
(here 1.0; the limit of 2 leaves room for a busy machine)."""
import pytest

pytestmark = pytest.mark.gpu


def test_cost_per_cell_of_an_iteration(cuda_lib):
    from paper_1410_1914_gb300 import Solver, structures
    cost = {}
    for edge in (64, 160):
        shape = (edge, edge + 1, edge - 1)
        s = Solver(shape, storage="fp32pop", dx_m=2e-9, knudsen=1, T_K=353.0, bc_in=0, bc_out=0, c_in=1.0, c_out=0.0)
        s.set_structure(structures.pt_cl(shape, 5, 0.45, 0.188743))
        best = float("inf")
        for _ in range(3):
            s.init()
            a = s.solve_steady_lines(tol=1e-30, max_iter=40, restart=40, cg_tol=0.5)   # exactly 40 iterations
            assert a["iterations"] == 40
            best = min(best, a["seconds"])
        cost[edge] = best / s.fluxes()["n_active"]
        s.close()
    assert cost[160] < 2.0 * cost[64], cost
