"""The tensor-core fit when one of its bounded waits runs out: the call comes
back with what its contract says, and nothing outside its own buffers is
written.  The waits are made to run out by their limit; the products themselves
finish as always."""
import ctypes as C

import numpy as np
import pytest

from paper_2301_05780_gb300 import pdds, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _data(n):
    g = torch.Generator(device="cuda").manual_seed(3)
    xy = torch.rand(n, 2, generator=g, device="cuda") * 2 - 1
    return xy, torch.sin(3 * xy[:, 0]) * torch.cos(2 * xy[:, 1])


DEFAULT = 2_000_000_000


def _fit(n, steps, **limits):
    """theta and the losses of the fit with the given wait limits (ns)."""
    f = pdds.lib().pdds_internal_mlp_train_tc
    f.restype = C.c_int
    f.argtypes = [C.c_void_p] * 3 + [C.c_int64, C.c_int32, C.c_double, C.c_void_p, C.c_void_p] + [C.c_uint64] * 2
    xy, t = _data(n)
    theta = torch.tensor(W.mlp_init(), dtype=torch.float32, device="cuda")
    loss = np.zeros(steps + 1)
    loss[steps] = 7.0
    st = f(theta.data_ptr(), xy.data_ptr(), t.data_ptr(), n, steps, 3e-3,
           loss.ctypes.data_as(C.c_void_p), None, limits.get("mma_ns", DEFAULT),
           limits.get("barrier_ns", DEFAULT))
    assert st == pdds.PDDS_OK
    assert loss[steps] == 7.0
    return theta.cpu().numpy(), loss[:steps]


# one tile; fewer tiles than SMs; more than two per SM
@pytest.mark.parametrize("n,steps", [(100, 1), (5_000, 20), (100_000, 5)])
def test_product_wait_that_runs_out_voids_that_steps_loss_only(n, steps):
    theta, loss = _fit(n, steps, mma_ns=0)
    assert np.isnan(loss).all()
    # the products finished within the second wait, so the steps themselves were
    # right: theta as without the timeouts, within the spread of FP32 sums in
    # arrival order (each Adam step moves a parameter by at most about lr)
    want, wloss = _fit(n, steps)
    assert np.isfinite(wloss).all()
    assert np.abs(theta - want).max() <= 2 * 3e-3 * steps
    assert np.linalg.norm(theta - want) <= 1e-2 * np.linalg.norm(want)


@pytest.mark.parametrize("n,steps", [(100, 1), (100, 40), (5_000, 1), (5_000, 40), (30_000, 40)])
def test_barrier_wait_that_runs_out_does_not_lose_the_fit(n, steps):
    """A CTA that would have to wait at the grid barrier gives up at once: the run
    is taken again launch by launch, from the parameters as they were given."""
    theta, loss = _fit(n, steps, barrier_ns=0)
    want, wloss = _fit(n, steps)
    assert np.isfinite(loss).all()
    # the first loss is that of the given parameters (BF16 products, FP64 sum in
    # arrival order)
    assert abs(loss[0] - wloss[0]) <= 1e-9 * wloss[0]
    assert loss[-1] <= loss[0]
    assert np.abs(theta - want).max() <= 2 * 3e-3 * steps
    assert np.linalg.norm(theta - want) <= 1e-2 * np.linalg.norm(want)
