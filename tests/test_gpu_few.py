"""Expansions that admit a few candidates insert them one by one (compact
kernel, out-degree 32): the same searches as the general kernel's on batches
large enough to meet every case -- candidates at either end of the beam,
pushed past the cut by a smaller one, already there -- and the same counts of
inserted candidates, which the learned stop's features 7 and 10 carry."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gpu_index(tmp_path_factory, lib_built):
    from paper_2411_12229_gb300 import index_builder as ib
    from paper_2411_12229_gb300 import synth
    from paper_2411_12229_gb300.api import Index
    w = synth.small(synth.BATCHED_1M_D128, 20_000, 4_000)
    p = tmp_path_factory.mktemp("few") / "few.sqg"
    ib.build_index(p, synth.base(w), 32, device=0, init="random", iterations=2, ef_build=64)
    return Index(p, 0), torch.from_numpy(synth.queries(w)).cuda()


@pytest.mark.parametrize("k,ef", [(1, 1), (1, 2), (2, 3), (10, 31), (10, 32), (10, 33), (10, 64), (10, 65), (10, 96),
                                  (100, 128), (10, 129), (100, 200), (128, 256)])
def test_equals_the_general_kernel(gpu_index, k, ef):
    ix, q = gpu_index
    a = ix.search(q, k, ef, stats=True, kernel=2)
    b = ix.search(q, k, ef, stats=True, kernel=1)
    assert all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("k,ef", [(1, 4), (10, 20), (10, 64), (10, 100), (10, 180), (64, 100)])
@pytest.mark.parametrize("feature", [7, 10])
def test_stop_sees_the_inserted_candidates(gpu_index, k, ef, feature):
    """A network that passes one feature through, stopping on thresholds
    between its possible values: one candidate more or less moves the stop."""
    ix, q = gpu_index
    p = np.zeros(5313, np.float32)
    p[:1024].reshape(64, 16)[0, feature] = -1.0  # relu(1 - f): falls with the feature
    p[1024:1088][0] = 1.0
    p[1088:5184].reshape(64, 64)[0, 0] = 1.0
    p[5248:5312][0] = 1.0
    net = torch.from_numpy(p).cuda()
    for thr in (1 - 0.5 / 32, 1 - 1.5 / 32, 1 - 2.5 / 32):  # f below 0.5, 1.5, 2.5 candidates of 32
        kw = dict(stats=True, stop_mlp=net, stop_logit=float(thr), stop_every=1)
        a = ix.search(q, k, ef, kernel=2, **kw)
        b = ix.search(q, k, ef, kernel=1, **kw)
        assert all(torch.equal(x, y) for x, y in zip(a, b))
        assert bool((a[2][:, 1] & 2).any())  # the stop fired
