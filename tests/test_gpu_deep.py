"""The deep-beam search kernel (search_deep.cuh: a small front merged at every
expansion, a main part merged when the front is full) against the general
kernel and the oracle: ids, distances, hop counts, status bits and the
expansion order identical, at the edges of the front (ef 64 / 65, 128 / 129),
of the 32-entry window and of the main part, on the shapes of the workloads."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gpu_tiny(tiny_index):
    from paper_2411_12229_gb300.api import Index
    p, x, q = tiny_index
    return Index(p, 0), p, q


def same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))


def check(ix, O, q, k, ef, oracle_queries=4, **kw):
    """Default dispatch = general kernel, with and without the path; the
    first queries = the oracle."""
    qd = torch.from_numpy(q).cuda()
    ids, dists, st = ix.search(qd, k, ef, stats=True, **kw)
    g = ix.search(qd, k, ef, stats=True, kernel=1, **kw)
    assert same((ids, dists, st), g)
    cap = 4 * ef + 64
    t = ix.search_trace(qd, k, ef, None, 0, path_cap=cap, **kw)
    tg = ix.search_trace(qd, k, ef, None, 0, path_cap=cap, kernel=1, **kw)
    assert same(t[:3], g) and same(tg[:3], g) and torch.equal(t[-1], tg[-1])
    short = ix.search_trace(qd, k, ef, None, 0, path_cap=7, **kw)  # path_cap below the hops
    assert torch.equal(short[-1], tg[-1][:, :7])
    okw = {"eps0": kw.get("eps0", 0.0)}
    if kw.get("hop_cap"):
        okw["hop_cap"] = kw["hop_cap"]
    for i in range(min(oracle_queries, q.shape[0])):
        oi, od, oh, os_ = O.search(q[i], k, ef, **okw)
        np.testing.assert_array_equal(ids[i].cpu().numpy().view(np.uint32), oi)
        np.testing.assert_array_equal(dists[i].cpu().numpy(), od)
        assert tuple(st[i].tolist()) == (oh, os_)


@pytest.mark.parametrize("k,ef", [(1, 1), (1, 2), (5, 63), (10, 64), (10, 65), (1, 66), (32, 95), (33, 96), (10, 97),
                                  (128, 128), (100, 129), (10, 257), (100, 300), (64, 400), (128, 511), (1, 512),
                                  (100, 1025), (10, 2048)])
def test_deep_on_tiny(gpu_tiny, oracle_mod, k, ef):
    ix, p, q = gpu_tiny
    check(ix, oracle_mod.Index(p), q, k, ef)


@pytest.mark.parametrize("kw", [{"eps0": 1.9}, {"hop_cap": 1}, {"hop_cap": 30}, {"hop_cap": 100},
                                {"visited_smem_log2": 5}, {"visited_smem_log2": 12}, {"warps_per_block": 1},
                                {"rotation": 2}])
def test_deep_options(gpu_tiny, oracle_mod, kw):
    ix, p, q = gpu_tiny
    check(ix, oracle_mod.Index(p), q, 40, 300, **kw)


@pytest.mark.parametrize("k,ef", [(10, 60), (10, 130), (100, 200), (128, 400), (1, 900)])
def test_deep_shapes(shaped_index_file, oracle_mod, k, ef):
    from paper_2411_12229_gb300.api import Index
    p, _, q = shaped_index_file
    check(Index(p, 0), oracle_mod.Index(p), q, k, ef)


def test_deep_out_degree_64(tiny_index_r64, oracle_mod):
    from paper_2411_12229_gb300.api import Index
    p, _, q = tiny_index_r64
    ix, O = Index(p, 0), oracle_mod.Index(p)
    for k, ef in ((10, 127), (10, 128), (10, 129), (100, 300), (32, 700)):
        check(ix, O, q, k, ef)


def test_deep_duplicate_vectors_and_ties(tmp_path, lib_built, oracle_mod):
    """Repeated vectors: equal keys with different ids, and identical
    (key, id) pairs reached from identical vertices, in front and main part."""
    from paper_2411_12229_gb300 import index_builder as ib
    from paper_2411_12229_gb300.api import Index
    g = np.random.default_rng(3)
    x = np.repeat(g.standard_normal((150, 64)).astype(np.float32), 8, axis=0)
    x[::3] += 1e-3 * g.standard_normal((400, 64)).astype(np.float32)
    p = tmp_path / "dup.sqg"
    ib.build_index(p, x, 32)
    q = (x[g.integers(0, 1200, 24)] + 0.05 * g.standard_normal((24, 64))).astype(np.float32)
    ix, O = Index(p, 0), oracle_mod.Index(p)
    for k, ef in ((10, 80), (40, 140), (100, 257), (100, 600)):
        check(ix, O, q, k, ef, oracle_queries=8)


def test_deep_mixed_batch(gpu_tiny):
    """Per-query k and ef from one to past the front in one launch, invalid
    pairs among them."""
    ix, _, q = gpu_tiny
    qd = torch.from_numpy(np.concatenate([q] * 8)).cuda()
    g = np.random.default_rng(5)
    n = qd.shape[0]
    k = g.choice([1, 10, 100], n).astype(np.int32)
    ef = (k * g.integers(1, 9, n)).astype(np.int32)
    k[5], ef[9], ef[11] = 0, k[9] - 1, 801
    kt, et = torch.from_numpy(k).cuda(), torch.from_numpy(ef).cuda()
    a = ix.search(qd, kt, et, stats=True, max_k=100, max_ef=800)
    b = ix.search(qd, kt, et, stats=True, max_k=100, max_ef=800, kernel=1)
    assert same(a, b)


def test_least_workspace_still_serves(tmp_path, lib_built):
    """A workspace (or the fixed scratch) that holds the general kernel's
    visited tables but not the deep kernel's, whose build for d <= 512 keeps
    more warps resident: the search takes the general kernel, not an error."""
    from paper_2411_12229_gb300 import _binding as B
    from paper_2411_12229_gb300 import index_builder as ib
    from paper_2411_12229_gb300 import synth
    from paper_2411_12229_gb300.api import Index
    w = synth.small(synth.HIGHDIM_1M_D960.with_(d=512), 1500, 2400)
    p = tmp_path / "d512.sqg"
    ib.build_index(p, synth.base(w), 32)
    ix, q = Index(p, 0), torch.from_numpy(synth.queries(w)).cuda()
    k, ef, nq = 10, 300, q.shape[0]
    least, full = ix.workspace_size(nq, k, ef, kernel=1), ix.workspace_size(nq, k, ef)
    assert full > least
    ref = ix.search(q, k, ef, kernel=1)
    for size in (least, full):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        assert same(ix.search(q, k, ef, workspace=ws), ref)
    with pytest.raises(B.SqgError):
        ix.search(q, k, ef, workspace=torch.empty(least - 256, dtype=torch.uint8, device="cuda"))
    # the fixed scratch: the most queries whose least plan fits it
    limit = B.lib().sqg_noalloc_scratch_bytes()
    n = max(m for m in range(100, nq + 1, 50) if ix.workspace_size(m, k, ef, kernel=1) + 32768 <= limit)
    kt, et = (torch.full((n,), v, dtype=torch.int32, device="cuda") for v in (k, ef))
    ids, d = torch.empty(n * k, dtype=torch.int32, device="cuda"), torch.empty(n * k, device="cuda")
    rc = B.lib().sqg_search_noalloc(ix.handle, q.data_ptr(), n, kt.data_ptr(), et.data_ptr(), k, ef, ids.data_ptr(),
                                    d.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert rc == 0 and torch.equal(ids.view(n, k), ref[0][:n]) and torch.equal(d.view(n, k), ref[1][:n])


@pytest.mark.parametrize("nq", [1, 3, 64, 700])
def test_tables_of_a_resident_batch(gpu_tiny, nq):
    """Batches whose queries are all resident take larger visited tables: the
    searches of any batch size are the same."""
    ix, _, q = gpu_tiny
    qd = torch.from_numpy(np.concatenate([q] * 160)).cuda()  # past the resident warps: the small tables
    for k, ef in ((10, 64), (100, 160), (64, 400), (10, 1200)):
        ids, dists, st = ix.search(qd, k, ef, stats=True)
        assert same(ix.search(qd[:nq], k, ef, stats=True), (ids[:nq], dists[:nq], st[:nq]))
