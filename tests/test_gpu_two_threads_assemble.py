"""Contexts of one coefficient set share their path kernel, and with it the
kernel's shared-memory limit on the device: two threads that assemble their own
problems must not see each other's launch plans.  The problems are the ones whose
plan is not the first size it asks about (three stages per CTA), assembled next
to each other many times; every result is the serial one."""
import threading

import pytest

from paper_2301_05780_gb300 import pdds, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _finish(w):
    w.grid["ext"] = W.stencil_extension(w.grid, w.sigma_bounds[1], w.dt)
    w.k_max = W.step_cap(w.grid, w.sigma_bounds[0], w.dt)
    return w


def _table():
    # 1,729 knots >= 3 stages x 2 CTAs x 152 SMs, >= 512 paths each
    g = dict(x0=0.0, x1=1.0, y0=0.0, y1=1.0, Hx=8, Hy=8, m=16, ext=0)
    w = W.Workload("table", g, W.COEF_TABLE, params=(1.0, 0.5), n_paths=512, dt=1e-5, seed=11,
                   sigma_bounds=(1.1, 1.72))
    w.tables = W.config4_tables(257, 257)
    return _finish(w)


def _shifted():
    # 11,761 knots >= 3 stages x 18 CTAs x 152 SMs
    g = dict(x0=0.0, x1=1.0, y0=0.0, y1=1.0, Hx=20, Hy=20, m=16, ext=0)
    return _finish(W.Workload("gm", g, W.COEF_MANUFACTURED, n_paths=100, dt=1e-6, seed=12,
                              sigma_bounds=(2 ** 0.5, 2 ** 0.5)))


@pytest.mark.parametrize("make,scheme", [(_table, pdds.PDDS_SCHEME_EM), (_shifted, pdds.PDDS_SCHEME_GM)],
                         ids=["table", "gm"])
def test_threads_do_not_disturb_each_others_launches(make, scheme):
    probs = [pdds.Problem(make()) for _ in range(2)]
    want = []
    for P in probs:
        pdds.pdds_set_scheme(P.ctx, scheme)
        P.assemble()
        want.append(P.val.clone())
    torch.cuda.synchronize()
    bad = []

    def work(i):
        P, s = probs[i], torch.cuda.Stream()
        try:
            for _ in range(200):
                P.assemble(stream=s)
            s.synchronize()
            if pdds.pdds_stats(P.ctx)["device_error"] != 0 or not torch.equal(P.val, want[i]):
                bad.append((i, "result"))
        except Exception as e:
            bad.append((i, repr(e)))

    ts = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not bad, bad
