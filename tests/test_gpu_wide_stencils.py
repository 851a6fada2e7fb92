"""Stencils so wide that a larger unit ring needs all of a CTA's shared memory: the
launch plan then keeps the ring that fits instead of refusing the assembly."""
import pytest

from paper_2301_05780_gb300 import pdds, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# A corner knot of a 4 x 4 decomposition has 8 m + 4 + 8 ext accumulator slots.
# With the tcgen05 network (34,816 bytes) four stages of 6,113 to 6,128 slots
# (49,408 bytes each) come to 232,448 bytes, the whole of a CTA's limit.
@pytest.mark.parametrize("m", [762, 763, 764, 765])
def test_network_assembly_with_stages_at_the_shared_memory_limit(m):
    g = dict(x0=0.0, x1=1.0, y0=0.0, y1=1.0, Hx=4, Hy=4, m=m, ext=1)
    w = W.Workload("wide", g, W.COEF_LAPLACE_EXPSIN, n_paths=1, dt=1e-3, seed=5)
    w.k_max = W.step_cap(g, 2 ** 0.5, 1e-3)
    P = pdds.Problem(w)
    pdds.pdds_set_control_variate(P.ctx, torch.tensor(W.mlp_init(), dtype=torch.float32, device="cuda"))
    P.assemble()
    st = pdds.pdds_stats(P.ctx)
    assert st["device_error"] == 0 and st["paths"] == P.n
    assert torch.isfinite(P.b).all() and torch.isfinite(P.val).all()
