"""Device memory of the GPU adjust step: no more than the arrays that are
alive together need -- the reverse lists at their real length, the rows in
the candidate ids' place -- with room behind the rows for the reverse lists
and without; the rows are the host's either way."""

import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def build(x, cand, R, device):
    from paper_2411_12229_gb300 import index_builder as ib
    return ib.build_graph(x, cand, R, 0, 7, 0, device, True)


@pytest.mark.parametrize("L", [40, 100])
def test_memory_of_a_build(lib_built, L):
    n, d, R = 400_000, 32, 32
    g = np.random.default_rng(L)
    x = g.standard_normal((n, d), dtype=np.float32)
    cand = g.integers(0, n, (n, L), dtype=np.uint32)
    build(x[:1000], cand[:1000] % 1000, R, 0)  # the kernels are loaded
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    least, done = [before], threading.Event()

    def watch():
        while not done.is_set():
            least[0] = min(least[0], torch.cuda.mem_get_info()[0])

    t = threading.Thread(target=watch)
    t.start()
    try:
        stats = build(x, cand, R, 0)[1]
    finally:
        done.set()
        t.join()
    # data, candidate ids, own lists, kept edges and refined lists, counts and
    # flags, offsets, reverse lists
    row = 4 * d + 4 * L + 8 * L + 2 * 8 * R + 4 * 4 + 8 + 8 * stats["avg_nsg_degree"]
    assert 0.5 * n * row < before - least[0] < n * row + (24 << 20)  # (the driver's granules)


@pytest.mark.parametrize("L", [20, 33, 40, 70, 120])
def test_rows_where_the_arrays_share_memory(lib_built, L):
    g = np.random.default_rng(L)
    x = g.standard_normal((3000, 64)).astype(np.float32)
    cand = g.integers(0, 3000, (3000, L)).astype(np.uint32)
    cand[:, 0] = 17  # a hub: more reverse candidates than a warp's lists hold
    h, hs = build(x, cand, 32, None)
    d, ds = build(x, cand, 32, 0)
    np.testing.assert_array_equal(d, h)
    assert all(ds[k] == hs[k] for k in hs)
