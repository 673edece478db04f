"""A search on another stream than torch's current one, without any order of
the caller's: the padding, copies and fills that the call itself makes, and
tensors that the current stream is still producing, are read when they are
there, and none of their memory is handed out again before the search is
done."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LATE = 40_000_000  # cycles (about 20 ms) that a stream is held back


@pytest.fixture(scope="module", params=["fjlt", "dense"])
def index(request, tmp_path_factory, lib_built):
    """(index, queries): a fast-JLT index of 96 columns padded to 128, a dense one of 128."""
    from paper_2411_12229_gb300 import index_builder as ib
    from paper_2411_12229_gb300 import synth
    from paper_2411_12229_gb300.api import Index
    w = synth.small(synth.BATCHED_1M_D128.with_(d=96 if request.param == "fjlt" else 128), 1500, 300)
    p = tmp_path_factory.mktemp(request.param) / "i.sqg"
    ib.build_index(p, synth.base(w), 32, rotation=request.param)
    return Index(p, 0), torch.from_numpy(synth.queries(w)).cuda()


class Handle:
    """A stream of another library: an object with a ``cuda_stream``."""

    def __init__(self, s):
        self.cuda_stream = s.cuda_stream


def forms(nq):
    t = lambda v: torch.full((nq,), v, dtype=torch.int32, device="cuda")  # noqa: E731
    return {"numbers": (10, 64), "arrays": (np.full(nq, 10), np.full(nq, 64)), "tensors": (t(10), t(64)),
            "one of each": (10, t(64)), "k per query": (t(10), 64)}


@pytest.mark.parametrize("form", ["numbers", "arrays", "tensors", "one of each", "k per query"])
@pytest.mark.parametrize("strided", [False, True])
@pytest.mark.parametrize("foreign", [False, True])
def test_queries_of_the_current_stream(index, form, strided, foreign):
    ix, q = index
    nq = q.shape[0]
    k, ef = forms(nq)[form]
    ref = ix.search(q, k, ef, stats=True)
    late = torch.zeros((q.shape[1], nq), device="cuda").t() if strided else torch.zeros_like(q)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(LATE)
    late.copy_(q)  # still to come when the search is called
    got = ix.search(late, k, ef, stats=True, stream=Handle(s) if foreign else s)
    s.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, ref))


@pytest.mark.parametrize("form", ["numbers", "k per query"])
def test_memory_is_kept_until_the_search_is_done(index, form):
    """The search is held back while the caller lets go of everything and the
    current stream writes over what it is given."""
    ix, q = index
    nq = q.shape[0]
    k, ef = forms(nq)[form]
    ref = [r.clone() for r in ix.search(q, k, ef)]
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        torch.cuda._sleep(LATE)
    ids, dists = ix.search(torch.cat([q, q], 1)[:, :q.shape[1]], k, ef, stream=s)  # strided, and let go of
    trash = [torch.full((nq, c), 7.0, device="cuda") for c in (1, 10, q.shape[1], ix.d, 2 * q.shape[1])]
    s.synchronize()
    torch.cuda.synchronize()
    assert torch.equal(ids, ref[0]) and torch.equal(dists, ref[1])
    assert all(bool((t == 7.0).all()) for t in trash)


def test_traces_on_a_side_stream(index):
    ix, q = index
    ref = [None if t is None else t.clone() for t in ix.search_trace(q, 10, 64, None, 0, path_cap=100)]
    late = torch.zeros((q.shape[1], q.shape[0]), device="cuda").t()
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(LATE)
    late.copy_(q)
    got = ix.search_trace(late, 10, 64, None, 0, path_cap=100, stream=s)
    s.synchronize()
    for a, b in zip(got, ref):
        assert (a is None and b is None) or torch.equal(a, b)


def test_captured_with_a_side_stream(index):
    """Both streams in one capture: the search is ordered after the copy that
    the capture holds, at every replay."""
    ix, q = index
    ref = ix.search(q, 10, 64)
    ref = [r.clone() for r in ref]
    src, buf = torch.zeros_like(q), torch.zeros_like(q)
    out = (torch.empty(10 * len(q), dtype=torch.int32, device="cuda"), torch.empty(10 * len(q), device="cuda"))
    ws = torch.empty(ix.workspace_size(len(q), 10, 64), dtype=torch.uint8, device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        s.wait_stream(torch.cuda.current_stream())
        buf.copy_(src)
        ix.search(buf, 10, 64, out=out, workspace=ws, stream=s)
        torch.cuda.current_stream().wait_stream(s)
    src.copy_(q)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out[0].view(-1, 10), ref[0]) and torch.equal(out[1].view(-1, 10), ref[1])
