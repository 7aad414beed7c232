"""A caller's allocator (cl_params.alloc) promises no alignment beyond that of a
double: the calls that took such buffers give the results that they give with
the library's own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


class _Odd:
    """Allocations that start 8 bytes past a 256-byte boundary."""

    def __init__(self):
        import torch
        from paper_1410_1914_gb300 import _lib as L
        self.held = {}

        def alloc(n, stream, ctx):
            t = torch.empty(int(n) + 8, dtype=torch.uint8, device="cuda")
            assert t.data_ptr() % 256 == 0
            self.held[t.data_ptr() + 8] = t
            return t.data_ptr() + 8

        def free(ptr, n, stream, ctx):
            del self.held[ptr]

        self.alloc, self.free = L.cl_alloc_fn(alloc), L.cl_free_fn(free)


def _run(odd, storage, lattice, go, shape):
    from paper_1410_1914_gb300 import Solver, structures
    kw = dict(alloc=odd.alloc, free=odd.free) if odd else {}
    s = Solver(shape, storage=storage, lattice=lattice, dx_m=2e-9, knudsen=1, T_K=353.0, bc_in=0, bc_out=0, c_in=1.0,
               c_out=0.0, k_ms=1e3, react_rule=1, check_every=20, **kw)
    s.set_structure(structures.pt_cl(shape, 5, 0.45, 0.188743))
    info = go(s)
    out = (s.populations(), s.fluxes(), info)
    s.close()
    if odd:
        assert not odd.held   # everything was given back by the address that was handed out
    return out


def _same(storage, lattice, go, shape=(12, 13, 41)):
    (a, fa, ia), (b, fb, ib) = (_run(odd, storage, lattice, go, shape) for odd in (None, _Odd()))
    np.testing.assert_array_equal(a, b)
    assert fa == fb
    if ia:
        ia.pop("seconds"), ib.pop("seconds")
        assert ia == ib


@pytest.mark.parametrize("lattice", ["d3q7", "d3q19"])
def test_krylov_solve_with_buffers_of_eight_byte_alignment(cuda_lib, lattice):
    _same("fp32pop", lattice, lambda s: s.solve_krylov_dsa(tol=1e-7, max_iter=400, max_steps=20))


@pytest.mark.parametrize("storage", ["fp32", "fp16dev"])
def test_d3q19_step_with_buffers_of_eight_byte_alignment(cuda_lib, storage):
    _same(storage, "d3q19", lambda s: s.solve_budget(40))
