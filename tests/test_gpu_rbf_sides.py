"""RBF exits on stencils around the warp's passes (32 knots a pass, three passes
side by side in the assembly kernel, one in the records kernel): both kernels
deposit the same fixed-point weights, so G is the same bit for bit."""
import math

import numpy as np
import pytest

from paper_2301_05780_gb300 import pdds, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [2, 15, 16, 31, 47, 48, 63, 100])
def test_assembly_and_records_kernels_deposit_the_same_weights(m):
    w = W.config2().scaled(n_paths=40, dt=2e-4)
    w.grid = dict(w.grid, Hx=3, Hy=2, m=m, ext=1)   # stencils of m + 1 .. 2 m + 3 knots
    w.k_max = W.step_cap(w.grid, math.sqrt(2), w.dt)
    P = pdds.Problem(w)
    pdds.pdds_set_interpolation(P.ctx, pdds.PDDS_INTERP_RBF, 1.5 / (3 * m))
    P.assemble()
    val, b = P.val.cpu().numpy(), P.b.cpu().numpy()
    P.assemble(records=P.records_buffer())
    assert pdds.pdds_stats(P.ctx)["device_error"] == 0
    assert np.array_equal(val, P.val.cpu().numpy())
    # b: FP64 sums of 40 shares of order one, each of up to 2 m + 3 terms, in any order
    assert np.abs(b - P.b.cpu().numpy()).max() <= 300 * 2.0 ** -52 * max(1.0, np.abs(b).max())
    P.close()
