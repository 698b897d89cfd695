"""The network's gradient kernel at the edges of its slices (64 rows, 8 per CTA)
and of the fused reduction (up to 64 slices in one launch), for the smallest
and largest ladder, against the oracle's FP64 back-propagation.

Tolerance: a gradient entry is a sum over the m rows of products of fp32 dot
products of length <= 64 of O(1) operands, summed 64 rows at a time: an error
of at most (64 + m / 64 + 64) 2^-24 < 2e-5 of the sum of its terms'
magnitudes, which is below 5 times the largest entry: 1e-4 of the largest
entry plus 1e-7.  The loss, a mean of m such rows: 1e-5 relative."""
import numpy as np
import pytest

from oracle import jag_mlp as M

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
jag = pytest.importorskip("paper_2602_10258_gb300.jag")


@pytest.mark.parametrize("nl", [1, 16])
@pytest.mark.parametrize("m", [7, 65, 4096, 4097])
def test_gradient_at_slice_edges(m, nl):
    rng = np.random.default_rng(m + nl)
    X = rng.standard_normal((m, 12)).astype(np.float32)
    y = rng.integers(0, nl, m).astype(np.int32)
    t = rng.uniform(0, 3, m).astype(np.float32)
    theta = M.init_params(nl, seed=2).astype(np.float32)
    loss, g = jag.mlp_loss_grad(nl, torch.from_numpy(theta).cuda(), torch.from_numpy(X).cuda(),
                                torch.from_numpy(y).cuda(), torch.from_numpy(t).cuda(), 0.5)
    ref = M.grad(theta.astype(np.float64), X, y, t, nl, 0.5)
    assert np.abs(g.cpu().numpy() - ref).max() <= 1e-4 * np.abs(ref).max() + 1e-7
    want = M.loss(theta.astype(np.float64), X, y, t, nl, 0.5)
    assert abs(float(loss.cpu()[0]) - want) <= 1e-5 * abs(want)


def test_training_in_one_step_is_the_gradient_step():
    """One mini-batch of more slices than the fused launch takes, and one of
    fewer: the first Adam step moves every parameter by lr * g / (|g| + eps'),
    so the signs of the two results follow the gradient."""
    nl, lr = 5, 1e-3
    for m in (200, 5000):
        rng = np.random.default_rng(m)
        X = torch.from_numpy(rng.standard_normal((m, 12)).astype(np.float32)).cuda()
        y = torch.from_numpy(rng.integers(0, nl, m).astype(np.int32)).cuda()
        t = torch.from_numpy(rng.uniform(0, 3, m).astype(np.float32)).cuda()
        theta = torch.from_numpy(M.init_params(nl, seed=5).astype(np.float32)).cuda()
        _, g = jag.mlp_loss_grad(nl, theta, X, y, t, 0.5)
        p = theta.clone()
        tr = jag.Trainer(nl, p)
        tr.run(X, y, t, epochs=1, batch=m, lr=lr, lam=0.5)
        # the moments after one step hold the gradient itself: m = 0.1 g, one fp32 rounding
        assert torch.equal(tr.m, 0.1 * g)
        big = g.abs() > 1e-4
        assert torch.equal(torch.sign(theta - p)[big], torch.sign(g)[big])
