"""The compact kernel's builds for launches of a few queries per SM and those
with adders in the estimates: batch sizes on both sides of the rule's line (8
queries per SM) give the same searches as the general kernel, at d of one and
two chunks with whole and partial groups of code words."""

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("d", [32, 64, 96, 128, 160, 224, 256])
def test_batch_sizes_and_dimensions(tmp_path, lib_built, d):
    from paper_2411_12229_gb300 import index_builder as ib
    from paper_2411_12229_gb300 import synth
    from paper_2411_12229_gb300.api import Index
    w = synth.small(synth.BATCHED_1M_D128.with_(d=d), 1500, 1300)
    p = tmp_path / "i.sqg"
    ib.build_index(p, synth.base(w), 32)
    ix, q = Index(p, 0), torch.from_numpy(synth.queries(w)).cuda()
    for k, ef in ((1, 1), (10, 64), (10, 128), (10, 200), (100, 100), (128, 256)):
        ref = ix.search(q, k, ef, stats=True, kernel=1)
        for nq in (1, 2, 130, 1216, 1217, 1300):
            for eps0 in (0.0,) if nq != 130 else (0.0, 1.9):
                r = ref if eps0 == 0.0 else ix.search(q, k, ef, stats=True, kernel=1, eps0=eps0)
                got = ix.search(q[:nq], k, ef, stats=True, kernel=2, eps0=eps0)
                assert all(torch.equal(a, b[:nq]) for a, b in zip(got, r))
