"""A context that is given twice to the batched end-to-end call has one set of
device buffers: its solves must not run side by side on them."""
import numpy as np
import pytest

from paper_2301_05780_gb300 import pdds, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [(0, 0), (0, 1, 0), (1, 0, 0, 1)])
def test_repeated_context_in_a_host_batch(order):
    # teams of several CTAs (833 knots, 5e4 nonzeros) and one CTA (29 knots)
    ws = [W.config2().scaled(n_paths=200), W.config2().scaled(n_paths=200)]
    ws[1].grid["Hx"] = ws[1].grid["Hy"] = 4
    probs = [pdds.Problem(w) for w in ws]
    P = [probs[i] for i in order]
    out = [dict(rp=torch.empty(p.n + 1, dtype=torch.int32), col=torch.empty(p.nnz, dtype=torch.int32),
                val=torch.empty(p.nnz, dtype=torch.float64), b=torch.empty(p.n, dtype=torch.float64),
                u=torch.empty(p.n, dtype=torch.float64)) for p in P]
    pick = lambda k: [o[k] for o in out]
    pdds.pdds_assemble_solve_batch_host([p.ctx for p in P], 200, ws[0].dt, ws[0].seed, 1e-12, 5000,
                                        pick("rp"), pick("col"), pick("val"), pick("b"), pick("u"))
    for p, o in zip(P, out):
        rp, col, val = o["rp"].numpy(), o["col"].numpy(), o["val"].numpy()
        Gu = np.add.reduceat(val * o["u"].numpy()[col], rp[:-1])
        b = o["b"].numpy()
        # every output is the solution of the system returned beside it
        assert np.linalg.norm(b - Gu) <= 1e-11 * np.linalg.norm(b)
    for i in range(len(P)):
        for j in range(i):
            if P[i] is P[j]:
                assert torch.equal(out[i]["u"], out[j]["u"])
