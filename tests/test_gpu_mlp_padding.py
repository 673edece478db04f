"""The rows that fill up the last tile of the stop network's gradient kernel
take no part in it: a network whose logit overflows at a zero input, and is
finite on every sample, has the loss and the gradient of the oracle's fp64."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 63, 64, 65, 1000])
def test_overflow_at_a_zero_input(lib_built, oracle_mod, n):
    from paper_2411_12229_gb300 import learned_stop as L
    g = np.random.default_rng(n)
    P = (0.3 * g.standard_normal(5313)).astype(np.float32)
    W1, W2 = P[:1024].reshape(64, 16), P[1088:5184].reshape(64, 64)
    # hidden unit 0 is 1e30 (1 - x[0]): 0 on every sample, 1e30 at a zero input,
    # and the second layer's unit 0 overflows from it
    W1[0], W1[0, 0], P[1024] = 0.0, -1e30, 1e30
    W2[0, 0], P[5248] = 1e30, 1.0
    x = g.standard_normal((n, 16)).astype(np.float32)
    x[:, 0] = 1.0
    y = (g.uniform(size=n) > 0.4).astype(np.float32)
    w = g.uniform(0.2, 3.0, size=n).astype(np.float32)
    loss, grad = L.grad(*(torch.from_numpy(a).cuda() for a in (P, x, y, w)))
    lref, gref = oracle_mod.mlp_loss_grad_f64(P.astype(np.float64), x, y, w)
    assert np.isfinite(lref) and np.isfinite(gref).all()
    # fp32 sums of n terms: the bounds of the other gradient tests
    assert float(loss) == pytest.approx(lref, rel=1e-4)
    assert np.abs(grad.cpu().numpy() - gref).max() <= 1e-4 * np.abs(gref).max() + 1e-7
