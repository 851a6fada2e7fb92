"""The tensor-core evaluation of v_theta over the edges of its tiling (128-point
tiles, one per SM before a CTA's second warpgroup gets one, four warpgroups per
CTA), against the FP64 network; and calls from several threads at once, which
share the library's kept scratch buffer."""
import threading

import numpy as np
import pytest

from paper_2301_05780_gb300 import pdds, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _net64(th, xy):
    """v and grad v in FP64 (2 -> 64 -> 64 -> 1, SiLU), and running error bounds of an
    FP32 evaluation: 2^-20 (sixteen FP32 roundings: a few ulp of the logistic and of
    each product) of the sums of the magnitudes that every result is made of, the
    inputs of a SiLU carried on with slope at most 1.1 (SiLU') and 0.5 (SiLU'')."""
    th = th.double()
    W1, b1, W2, b2, w3, b3 = (th[:128].view(64, 2), th[128:192], th[192:4288].view(64, 64),
                              th[4288:4352], th[4352:4416], th[4416])
    x = xy.double()
    a1 = x @ W1.T + b1
    s1 = torch.sigmoid(a1)
    h1 = a1 * s1
    a2 = h1 @ W2.T + b2
    s2 = torch.sigmoid(a2)
    p1, p2 = s1 * (1 + a1 * (1 - s1)), s2 * (1 + a2 * (1 - s2))
    g2 = w3 * p2
    d1 = (g2 @ W2) * p1
    v, g = (a2 * s2) @ w3 + b3, d1 @ W1
    # magnitudes, in units of the rounding
    m1 = x.abs() @ W1.abs().T + b1.abs()                       # a1
    mh = 1.1 * m1 + h1.abs()                                   # h1
    m2 = mh @ W2.abs().T + b2.abs()                            # a2
    mv = (1.1 * m2 + (a2 * s2).abs()) @ w3.abs() + b3.abs()
    mg2 = w3.abs() * (0.5 * m2 + p2.abs())                     # g2
    mg = ((mg2 @ W2.abs()) * p1.abs() + (g2.abs() @ W2.abs()) * (0.5 * m1 + p1.abs())) @ W1.abs()
    return v, g, 2.0 ** -20 * mv, 2.0 ** -20 * mg


def _points(n, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed + n)
    return torch.rand(n, 2, generator=g, device="cuda") * 3 - 1.5


@pytest.mark.parametrize("scale", [1.0, 40.0])   # 40: saturated units (e^-a overflows in FP32)
@pytest.mark.parametrize("tiles,extra", [(0, 1), (1, -1), (1, 0), (1, 1), (152, 1), (304, 0),
                                         (608, 127), (700, 3)])
def test_eval_tc_at_tile_edges(tiles, extra, scale):
    theta = torch.tensor(W.mlp_init(), dtype=torch.float32, device="cuda")
    theta[:192] *= scale
    xy = _points(128 * tiles + extra)
    v, g = pdds.pdds_mlp_eval_tc(theta, xy)
    v64, g64, bv, bg = _net64(theta, xy)
    assert ((v.double() - v64).abs() <= bv).all()
    assert ((g.double() - g64).abs() <= bg).all()


def test_calls_from_several_threads_give_the_serial_results():
    theta = torch.tensor(W.mlp_init(), dtype=torch.float32, device="cuda")
    xys = [_points(5000 + 777 * i, i) for i in range(4)]
    want = [pdds.pdds_mlp_eval_tc(theta, xy) for xy in xys]
    want16 = [pdds.pdds_mlp_eval(theta, xy) for xy in xys]
    bad = []

    def work(i):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(20):
                v, g = pdds.pdds_mlp_eval_tc(theta, xys[i], stream=s)
                w, h = pdds.pdds_mlp_eval(theta, xys[i], stream=s)
                s.synchronize()
                if not (torch.equal(v, want[i][0]) and torch.equal(g, want[i][1]) and
                        torch.equal(w, want16[i][0]) and torch.equal(h, want16[i][1])):
                    bad.append(i)

    torch.cuda.synchronize()
    ts = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not bad
