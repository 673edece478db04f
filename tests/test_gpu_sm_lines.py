"""The dispatch lines that follow the GPU's number of SMs, on the SMs of the
GPU at hand: searches of 8 queries per SM and one more (the build for few
queries), rotations on both sides of four 32 x 64 tiles per SM, gradients of
one tile per SM and one sample more."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("d", [96, 256])
def test_searches(tmp_path, lib_built, sms, d):
    from paper_2411_12229_gb300 import index_builder as ib
    from paper_2411_12229_gb300 import synth
    from paper_2411_12229_gb300.api import Index
    w = synth.small(synth.BATCHED_1M_D128.with_(d=d), 1000, 8 * sms + 1)
    p = tmp_path / "i.sqg"
    ib.build_index(p, synth.base(w), 32)
    ix, q = Index(p, 0), torch.from_numpy(synth.queries(w)).cuda()
    for k, ef in ((10, 64), (10, 128), (100, 200)):
        ref = ix.search(q, k, ef, stats=True, kernel=1)
        for nq in (8 * sms - 1, 8 * sms, 8 * sms + 1):
            got = ix.search(q[:nq], k, ef, stats=True, kernel=2)
            assert all(torch.equal(a, b[:nq]) for a, b in zip(got, ref))


@pytest.mark.parametrize("d", [32, 64, 96, 128, 160, 256, 480])
def test_rotations(tmp_path, lib_built, sms, d):
    """The staging of a tile changes no bit: batches on both sides of the line
    against the same rows in calls of eight."""
    from paper_2411_12229_gb300 import index_builder as ib
    from paper_2411_12229_gb300 import synth
    from paper_2411_12229_gb300.api import Index
    w = synth.small(synth.BATCHED_1M_D128.with_(d=d), 200, 1)
    p = tmp_path / "i.sqg"
    ib.build_index(p, synth.base(w), 32)
    ix = Index(p, 0)
    line = 32 * -(-4 * sms // -(-d // 64))  # the most queries below the line, and those of the tile before
    q = torch.randn((line + 64, d), device="cuda", generator=torch.Generator(device="cuda").manual_seed(d))
    rows = range(0, line + 64, max(8, line // 40 // 8 * 8))
    ref = {i: ix.prepare_queries(q[i:i + 8].contiguous()) for i in rows}
    for nq in (line - 32, line - 31, line, line + 33, line + 64):
        got = ix.prepare_queries(q[:nq].contiguous())
        for i in rows:
            if i + 8 <= nq:
                assert all(torch.equal(a[i:i + 8], b) for a, b in zip(got, ref[i]))


@pytest.mark.parametrize("more", [-1, 0, 1])
def test_gradients(lib_built, oracle_mod, sms, more):
    from paper_2411_12229_gb300 import learned_stop as L
    n = 64 * sms + more
    g = np.random.default_rng(n)
    P = (0.3 * g.standard_normal(5313)).astype(np.float32)
    x = g.standard_normal((n, 16)).astype(np.float32)
    y = (g.uniform(size=n) > 0.4).astype(np.float32)
    w = g.uniform(0.2, 3.0, size=n).astype(np.float32)
    loss, grad = L.grad(*(torch.from_numpy(a).cuda() for a in (P, x, y, w)))
    lref, gref = oracle_mod.mlp_loss_grad_f64(P.astype(np.float64), x, y, w)
    # fp32 sums of n terms: the bounds of the other gradient tests
    assert float(loss) == pytest.approx(lref, rel=1e-4)
    assert np.abs(grad.cpu().numpy() - gref).max() <= 1e-4 * np.abs(gref).max() + 1e-7
