"""The library's own launch shape where a kernel's units cost more than their
paths: tabulated coefficients (a tile per unit), kernels whose warps step
together (the network) or do not draw ahead.  The units stay as few as stated,
and the records are those of an explicit shape, bit for bit."""
import numpy as np
import pytest

from paper_2301_05780_gb300 import pdds, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SETS = {
    "manufactured": (W.COEF_MANUFACTURED, 0.0, 1.0, ()),
    "varsigma": (W.COEF_VARSIGMA, 0.0, 4.0, ()),
    "table": (W.COEF_TABLE, 0.0, 1.0, (1.0, 0.5)),
    "e1": (W.COEF_POISSON_E1, -100.0, 100.0, ()),
}


def _problem(coef, H, m, N, steps, cv=None, scheme=pdds.PDDS_SCHEME_EM, engine=None, rbf=False):
    cid, lo, hi, params = SETS[coef]
    L = (hi - lo) / H
    dt = 0.25 * L * L / (2.0 * steps)
    w = W.Workload(coef, dict(x0=lo, x1=hi, y0=lo, y1=hi, Hx=H, Hy=H, m=m, ext=3), cid, params=params,
                   n_paths=N, dt=dt, seed=31, sigma_bounds=(0.9, 1.9))
    w.k_max = W.step_cap(w.grid, 0.9, dt)
    if coef == "table":
        w.tables = W.config4_tables(16 * H + 1, 16 * H + 1)
    P = pdds.Problem(w)
    pdds.pdds_set_scheme(P.ctx, scheme)
    if rbf:
        pdds.pdds_set_interpolation(P.ctx, pdds.PDDS_INTERP_RBF, 2.0 * L / m)
    if cv == "table":
        t = torch.linspace(0, 3, 41, device="cuda")
        pdds.pdds_set_control_variate_grid(P.ctx, torch.stack([torch.sin(t[:, None] + t), torch.cos(t[:, None] * t)], -1)
                                           .contiguous())
    elif cv == "network":
        pdds.pdds_set_control_variate(P.ctx, torch.tensor(W.mlp_init(), dtype=torch.float32, device="cuda"))
        if engine is not None:
            pdds.pdds_set_network_engine(P.ctx, engine)
    return P


# (the knots of the smallest case exceed its CTAs, so that one unit per knot is all there can be)
@pytest.mark.parametrize("coef,cv,engine,N", [
    ("table", None, None, 30), ("table", "table", None, 30),
    ("e1", None, None, 30), ("manufactured", "network", None, 30), ("manufactured", "network", None, 300),
    ("manufactured", "network", pdds.NET_MMA_SYNC, 30)])
def test_few_paths_per_knot_stay_one_unit(coef, cv, engine, N):
    P = _problem(coef, 8, 8, N, 20.0, cv, engine=engine)
    P.assemble()
    st = pdds.pdds_stats(P.ctx)
    assert st["device_error"] == 0 and st["paths"] == P.n * N
    assert st["units"] == P.n


@pytest.mark.parametrize("scheme", [pdds.PDDS_SCHEME_EM, pdds.PDDS_SCHEME_GM], ids=["em", "gm"])
@pytest.mark.parametrize("coef,cv,rbf", [
    ("table", "table", False), ("e1", "table", False), ("e1", None, False), ("varsigma", "table", False),
    ("e1", "network", False), ("manufactured", "network", False), ("manufactured", None, True),
    ("varsigma", "table", True)])
@pytest.mark.parametrize("H,m,N,ragged", [(2, 7, 9, False), (3, 5, 1100, False), (3, 5, 700, True)])
def test_records_do_not_depend_on_the_shape(coef, cv, rbf, scheme, H, m, N, ragged):
    out = []
    for launch in (None, (256, 1, 4096, 4), (64, 0, 96, 2)):
        P = _problem(coef, H, m, N, 18.0, cv, scheme, rbf=rbf)
        if ragged:   # none, one, a few, and up to three times N
            r = np.random.default_rng(5)
            P.n_per_knot = torch.tensor(r.choice([0, 1, 7, N // 2, N, 3 * N], P.n), device="cuda")
        if launch:
            pdds.pdds_set_launch(P.ctx, *launch)
        rec = P.records_buffer()
        P.assemble(records=rec)
        st = pdds.pdds_stats(P.ctx)
        assert st["device_error"] == 0
        out.append((pdds.records_to_numpy(rec).copy(), P.val.cpu().numpy(), P.b.cpu().numpy()))
        P.close()
    for other in out[1:]:
        assert out[0][0].tobytes() == other[0].tobytes()
        assert np.array_equal(out[0][1], other[1])   # exact sums of fixed-point weights
        # b: FP64 sums of the same numbers in another order
        assert np.allclose(out[0][2], other[2], rtol=1e-12, atol=1e-12)


@pytest.mark.parametrize("coef,cv", [("e1", None), ("e1", "table"), ("table", "table"), ("manufactured", "table"),
                                     ("e1", "network")])
def test_calibration_does_not_depend_on_the_shape(coef, cv):
    mom = []
    for launch in (None, (128, 0, 64, 1), (256, 1, 4096, 8)):
        P = _problem(coef, 3, 6, 400, 25.0, cv)
        if launch:
            pdds.pdds_set_launch(P.ctx, *launch)
        u0 = torch.linspace(-1, 2, P.n, dtype=torch.float64, device="cuda")
        m = torch.empty(P.n, 8, dtype=torch.float64, device="cuda")
        pdds.pdds_calibrate(P.ctx, u0, m, P.w.n_paths, None, P.w.dt, P.w.seed)
        assert pdds.pdds_stats(P.ctx)["device_error"] == 0
        mom.append(m.cpu().numpy())
        P.close()
    assert np.array_equal(mom[0], mom[1]) and np.array_equal(mom[0], mom[2])
