"""A batch with one k and one ef passes them by value (sqg_search_uniform)
and takes its scratch from the handle's own pool: the same results as the
array form, on the caller's stream, from several threads, repeatedly."""

import threading

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gpu_tiny(tiny_index):
    from paper_2411_12229_gb300.api import Index
    p, _, q = tiny_index
    return Index(p, 0), q


@pytest.mark.parametrize("k,ef,kw", [(1, 1, {}), (10, 64, {}), (32, 128, {}), (100, 200, {}), (10, 300, {}),
                                     (256, 2048, {}), (10, 64, {"kernel": 1}), (10, 48, {"team": 16}),
                                     (10, 64, {"rotation": 2}), (10, 64, {"max_ef": 100}),
                                     (10, 64, {"multi_estimate": False})])
def test_by_value_equals_the_arrays(gpu_tiny, k, ef, kw):
    ix, q = gpu_tiny
    qd = torch.from_numpy(q).cuda()
    nq = qd.shape[0]
    kt = torch.full((nq,), k, dtype=torch.int32, device="cuda")
    et = torch.full((nq,), ef, dtype=torch.int32, device="cuda")
    ref = ix.search(qd, kt, et, stats=True, **{"max_k": k, "max_ef": ef, "uniform_k": k, **kw})
    for _ in range(3):  # the default pool first, then the handle's own
        got = ix.search(qd, k, ef, stats=True, **kw)
        for a, b in zip(ref, got):
            assert torch.equal(a, b)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    got = ix.search(qd, k, ef, stats=True, stream=s, **kw)
    s.synchronize()
    for a, b in zip(ref, got):
        assert torch.equal(a, b)


def test_refused_as_before(gpu_tiny):
    from paper_2411_12229_gb300 import _binding as B
    ix, q = gpu_tiny
    qd = torch.from_numpy(q).cuda()
    for k, ef in ((10, 5), (10, 2049), (B.MAX_K + 1, 300)):
        with pytest.raises(B.SqgError):
            ix.search(qd, k, ef)
    L = B.lib()
    out = torch.empty(10 * len(q), dtype=torch.int32, device="cuda")
    d = torch.empty(10 * len(q), device="cuda")
    args = (out.data_ptr(), d.data_ptr(), None, None, 0, None, None)
    for k, ef in ((0, 10), (10, 0), (257, 300)):
        assert L.sqg_search_uniform(ix.handle, qd.data_ptr(), len(q), k, ef, *args) == -1
    p = ix.params(uniform_k=5)
    assert L.sqg_search_uniform(ix.handle, qd.data_ptr(), len(q), 10, 64, out.data_ptr(), d.data_ptr(),
                                B.C.byref(p), None, 0, None, None) == -1


def test_threads_share_the_handles_pool(gpu_tiny):
    ix, q = gpu_tiny
    qd = torch.from_numpy(q).cuda()
    ref = ix.search(qd, 10, 64)
    bad = []

    def work():
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(20):
                ids, dists = ix.search(qd, 10, 64)
                s.synchronize()
                if not (torch.equal(ids, ref[0]) and torch.equal(dists, ref[1])):
                    bad.append(1)

    torch.cuda.synchronize()
    ts = [threading.Thread(target=work) for _ in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad
