"""The solve when a barrier between its CTAs is not met in time (other work on the
device can keep some of them from starting): the problem is solved again on one
CTA, from the right-hand side as it was given."""
import ctypes as C

import numpy as np
import pytest

from paper_2301_05780_gb300 import pdds
from test_gpu_solve_shapes import _system

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _solve(G, b, u, wait_ns):
    f = pdds.lib().pdds_internal_solve_noalloc
    f.restype = C.c_int
    f.argtypes = [C.c_void_p] * 3 + [C.c_double, C.c_int32, C.c_void_p, C.c_void_p, C.c_uint64]
    it = C.c_int32()
    g = pdds._csr_struct(G)
    st = f(C.byref(g), b.data_ptr(), u.data_ptr(), 1e-12, 1000, C.byref(it), None, wait_ns)
    assert st == pdds.PDDS_OK
    return it.value


# one CTA (nothing to wait for); teams of several
@pytest.mark.parametrize("n,per_row", [(255, 40), (1025, 260), (3001, 120)])
@pytest.mark.parametrize("in_place", [False, True])
def test_barrier_wait_that_runs_out_does_not_lose_the_solve(n, per_row, in_place):
    A, rp, col, val, b = _system(n, per_row, n)
    dev = lambda a: torch.tensor(a, device="cuda")
    G, bd = (dev(rp), dev(col), dev(val)), dev(b)
    u = bd if in_place else torch.full_like(bd, float("nan"))
    assert _solve(G, bd, u, 0) >= 1
    got = u.cpu().numpy()
    # the bounds of test_gpu_solve_shapes: stopped at 1e-12 ||b||, ||A^-1||_inf <= 10
    assert np.linalg.norm(b - A @ got) <= 1e-11 * np.linalg.norm(b)
    assert np.abs(got - np.linalg.solve(A, b)).max() <= 10 * 1e-11 * np.linalg.norm(b)
    if not in_place:   # and as without the timeout, within the same bound
        w = torch.empty_like(u)
        _solve(G, bd, w, 10**10)
        assert np.abs(got - w.cpu().numpy()).max() <= 20 * 1e-11 * np.linalg.norm(b)
