"""The path kernel's stepping variants and the library's own launch shape.

Few paths per warp (a small problem, or the end of any launch) are stepped with
normals that the idle lanes draw ahead, the step cap is tested per visit of the
step loop instead of per step, and the unit size follows the problem: none of
this may change a path.  Records of the library's choice of shape are compared
bit for bit with those of explicit shapes that fill every warp, and (K, side)
with the FP64 oracle's."""
import numpy as np
import pytest

from paper_2301_05780_gb300 import pdds, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SETS = {
    "laplace": (W.COEF_LAPLACE_EXPSIN, 0.0, 1.0, ()),
    "manufactured": (W.COEF_MANUFACTURED, 0.0, 1.0, ()),
    "varsigma": (W.COEF_VARSIGMA, 0.0, 4.0, ()),
    "table": (W.COEF_TABLE, 0.0, 1.0, (1.0, 0.5)),
    "constant": (W.COEF_CONSTANT, 0.0, 1.0, (1.3, 0.4, -0.2, -0.7, 0.3, 1.1)),
    "e1": (W.COEF_POISSON_E1, -100.0, 100.0, ()),
}


def _workload(coef, N, steps, k_max=0):
    cid, lo, hi, params = SETS[coef]
    H, m = 3, 5
    L = (hi - lo) / H
    dt = 0.25 * L * L / (2.0 * steps)
    w = W.Workload(coef, dict(x0=lo, x1=hi, y0=lo, y1=hi, Hx=H, Hy=H, m=m, ext=4), cid, params=params,
                   n_paths=N, dt=dt, seed=97, sigma_bounds=(0.9, 1.9))
    w.k_max = k_max or W.step_cap(w.grid, 0.9, dt)
    if coef == "table":
        s, c = W.config4_tables(33, 33)
        w.tables = (s, c)
    return w


def _records(w, scheme, launch=None, budgets=None):
    P = pdds.Problem(w)
    pdds.pdds_set_scheme(P.ctx, scheme)
    if launch is not None:
        pdds.pdds_set_launch(P.ctx, *launch)
    if budgets is not None:
        P.n_per_knot = torch.tensor(budgets, device="cuda")
    rec = P.records_buffer()
    P.assemble(records=rec)
    st = pdds.pdds_stats(P.ctx)
    assert st["device_error"] == 0
    out = pdds.records_to_numpy(rec).copy(), P.val.cpu().numpy(), P.b.cpu().numpy(), st
    P.close()
    return out


@pytest.mark.parametrize("scheme", [pdds.PDDS_SCHEME_EM, pdds.PDDS_SCHEME_GM], ids=["em", "gm"])
@pytest.mark.parametrize("coef", list(SETS))
@pytest.mark.parametrize("N,steps,k_max", [(1, 60.0, 0), (33, 60.0, 0), (700, 25.0, 0), (33, 60.0, 37)])
def test_launch_shape_never_changes_a_path(orc, coef, scheme, N, steps, k_max):
    w = _workload(coef, N, steps, k_max)
    a = _records(w, scheme)
    b = _records(w, scheme, launch=(512, 1, 16384, 1))
    assert a[0].tobytes() == b[0].tobytes()
    assert np.array_equal(a[1], b[1])      # fixed-point slot sums: exact in any order
    # b: FP64 sums of N shares in different orders
    scale = np.abs(a[0]["b_contrib"].astype(np.float64)).max() + 1e-300
    assert np.abs(a[2] - b[2]).max() <= 4 * N * 2.0 ** -53 * scale
    if k_max:
        assert (a[0]["side_flags"] >> 8 & 1).any() and a[0]["steps"].max() == k_max
    if N == 33:
        O = orc.Problem(w.grid, w.coef_id, w.params, *(w.tables or (None, None)))
        kw = {} if scheme == pdds.PDDS_SCHEME_EM else {"scheme": 1}
        o = O.assemble(w.n_paths, w.dt, w.seed, w.k_max, records=True, **kw)[3]
        same = (a[0]["steps"] == o["steps"]) & ((a[0]["side_flags"] & 0xFF) == o["side"])
        # FP32 positions against FP64 ones: the flip fraction the parity tests allow is
        # 1e-3 of the paths, here of about 2,000 (two)
        assert np.count_nonzero(~same) <= max(2, 1e-3 * len(same))


def test_ragged_budgets_choose_the_unit_size_on_the_device():
    w = _workload("manufactured", 0, 40.0)
    n = pdds.pdds_geometry_host(w.grid)[0].shape[0]
    for top in (3, 90, 40_000):
        N = np.random.default_rng(top).integers(0, top, n)
        N[0] = 0
        a = _records(w, pdds.PDDS_SCHEME_EM, budgets=N)
        b = _records(w, pdds.PDDS_SCHEME_EM, launch=(512, 1, 16384, 1), budgets=N)
        assert a[3]["paths"] == N.sum()
        assert a[0].tobytes() == b[0].tobytes() and np.array_equal(a[1], b[1])
