"""The stop network's gradient at the edges of the kernel's tiles (64 samples,
one block per SM, so several tiles per block from 64 x SMs on), with and
without the loss, and with a gradient buffer that is only 4-byte aligned,
against the oracle's fp64."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 63, 64, 65, 128, 8192, 64 * 152, 64 * 152 + 1, 20011])
@pytest.mark.parametrize("shift", [0, 1])
def test_gradient_over_tiles(lib_built, oracle_mod, n, shift):
    from paper_2411_12229_gb300 import _binding as B
    g = np.random.default_rng(n)
    P = (0.3 * g.standard_normal(5313)).astype(np.float32)
    x = g.standard_normal((n, 16)).astype(np.float32)
    y = (g.uniform(size=n) > 0.4).astype(np.float32)
    w = g.uniform(0.2, 3.0, size=n).astype(np.float32)
    d = [torch.from_numpy(a).cuda() for a in (P, x, y, w)]
    buf = torch.full((5313 + 8,), 7.0, device="cuda")
    grad, scratch, loss = buf[shift:shift + 5313], torch.empty(1, device="cuda"), torch.empty(1, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    for lp in (loss.data_ptr(), None):
        B.check(B.lib().sqg_mlp_grad(*(t.data_ptr() for t in d), n, grad.data_ptr(), lp, scratch.data_ptr(), s), "grad")
    lref, gref = oracle_mod.mlp_loss_grad_f64(P.astype(np.float64), x, y, w)
    # fp32 sums of n terms: the same bounds as the other gradient tests
    assert float(loss) == pytest.approx(lref, rel=1e-4)
    assert np.abs(grad.cpu().numpy() - gref).max() <= 1e-4 * np.abs(gref).max() + 1e-7
    rest = torch.cat([buf[:shift], buf[shift + 5313:]])
    assert bool((rest == 7.0).all())  # nothing outside the gradient is written
