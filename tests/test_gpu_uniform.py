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


def run_threads(jobs):
    """Each job in a thread of its own; their exceptions and False results."""
    bad = []

    def work(job):
        try:
            if not job():
                bad.append("wrong results")
        except Exception as e:  # noqa: BLE001
            bad.append(repr(e))

    torch.cuda.synchronize()
    ts = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    return bad


def searcher(ix, q, k, ef, reps, **kw):
    ref = ix.search(q, k, ef, **kw)

    def job():
        s = torch.cuda.Stream()
        ok = True
        with torch.cuda.stream(s):
            for _ in range(reps):
                got = ix.search(q, k, ef, **kw)
                s.synchronize()
                ok = ok and torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
        return ok

    return job


def test_threads_share_the_handles_pool(gpu_tiny):
    ix, q = gpu_tiny
    qd = torch.from_numpy(q).cuda()
    assert run_threads([searcher(ix, qd, 10, 64, 20) for _ in range(4)]) == []


def test_threads_with_different_shapes(gpu_tiny, shaped_index_file):
    """Batches whose kernels are the same but whose shared memory differs (batch
    size, ef, visited tables, block size), on two indexes at once: no thread's
    launch is refused."""
    from paper_2411_12229_gb300.api import Index
    ix, q = gpu_tiny
    q1 = torch.from_numpy(q).cuda()
    big = q1.repeat(200, 1)
    p, _, qs = shaped_index_file
    ix2, q2 = Index(p, 0), torch.from_numpy(qs).cuda()
    jobs = [searcher(ix, q1, 10, 64, 60), searcher(ix, big, 10, 64, 20), searcher(ix, q1, 10, 50, 60, visited_smem_log2=11),
            searcher(ix, q1, 10, 400, 40), searcher(ix, q1, 10, 900, 40), searcher(ix, q1, 10, 64, 60, kernel=1),
            searcher(ix2, q2, 10, 64, 60), searcher(ix2, q2, 10, 300, 40), searcher(ix, q1, 10, 64, 60, warps_per_block=1)]
    assert run_threads(jobs) == []
