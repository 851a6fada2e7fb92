"""The trainers' gradient reductions and the one-launch training run at their
edges: a gradient buffer that is not 16-byte aligned (added float by float, not
by fours), and point counts around a full tile and around one tile per SM (the
largest run that is a single cooperative launch)."""
import numpy as np
import pytest

from paper_2301_05780_gb300 import pdds, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _data(n):
    r = np.random.default_rng(n)
    xy = r.uniform(-1, 1, (n, 2))
    dev = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")
    return dev(xy), dev(np.sin(3 * xy[:, 0]) * xy[:, 1]), dev(W.mlp_init())


@pytest.mark.parametrize("engine", ["fp32", "tc"])
def test_unaligned_gradient_buffer(engine):
    xy, t, theta = _data(5000)
    _, want = pdds.pdds_mlp_loss_grad(theta, xy, t, engine=engine)
    fn = pdds.lib().pdds_mlp_loss_grad_tc if engine == "tc" else pdds.lib().pdds_mlp_loss_grad
    for shift in (1, 2, 3, 4):
        buf = torch.full((pdds.MLP_NPARAM + 8,), float("nan"), dtype=torch.float32, device="cuda")
        g = buf[shift:shift + pdds.MLP_NPARAM]
        loss = torch.empty(1, dtype=torch.float64, device="cuda")
        pdds._check(fn(theta.data_ptr(), xy.data_ptr(), t.data_ptr(), t.numel(), g.data_ptr(),
                       loss.data_ptr(), pdds._stream(None)))
        torch.cuda.synchronize()
        # the same products, FP32 sums of the CTAs' parts in any order: 79 parts of at most
        # the total's size
        assert (g - want).abs().max() <= 79 * 2.0 ** -23 * want.abs().max()
        assert torch.isnan(buf[:shift]).all() and torch.isnan(buf[shift + pdds.MLP_NPARAM:]).all()


@pytest.mark.parametrize("n", [1, 127, 128, 129, 152 * 128, 152 * 128 + 1])
def test_training_steps_follow_the_gradient(n):
    """Each loss of a run equals the loss of the gradient call at the parameters a shorter run
    ends with, whichever way the steps are launched."""
    xy, t, theta0 = _data(n)
    full = pdds.pdds_mlp_train(theta0.clone(), xy, t, steps=5, engine="tc")
    for k in range(5):
        th = theta0.clone()
        if k:
            short = pdds.pdds_mlp_train(th, xy, t, steps=k, engine="tc")
            # FP32 reductions in another order move theta by some 1e-7; the BF16 operands then
            # round differently at a few points: 2^-8 of their share
            assert np.abs(short - full[:k]).max() <= 1e-3 * full[0]
        loss, _ = pdds.pdds_mlp_loss_grad(th, xy, t, engine="tc")
        assert abs(loss.item() - full[k]) <= 1e-3 * full[0]
