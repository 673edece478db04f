"""The reachability flood of the GPU adjust step on graphs of many levels: a
chain has as many as it has vertices, and past a number of them the flood is
the host's.  The rows are the host build's on both sides of that number, over
several rounds of the repair, and a long chain costs what its edges do, not a
launch over all vertices for each."""

import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def chain(n, piece):
    """n points on a line, each with the three on either side as candidates
    within its piece: without the angle rule every vertex keeps its two
    neighbours."""
    x = np.zeros((n, 32), np.float32)
    x[:, 0] = np.arange(n)
    i = np.arange(n)[:, None]
    cand = i + np.array([-3, -2, -1, 1, 2, 3])
    cand[(cand < 0) | (cand >= n) | (cand // piece != i // piece)] = 0xFFFFFFFF
    return x, cand.astype(np.uint32)


def build(x, cand, entry, device):
    from paper_2411_12229_gb300 import index_builder as ib
    return ib.build_graph(x, cand, 32, entry, 7, 0, device, False)


@pytest.mark.parametrize("n", [60, 64, 65, 71, 72, 73, 80, 1000, 9000, 20000])
@pytest.mark.parametrize("pieces", [1, 3])
def test_rows_of_chains(lib_built, n, pieces):
    x, cand = chain(n, -(-n // pieces))
    for entry in (0, n // 2):
        h, hs = build(x, cand, entry, None)
        d, ds = build(x, cand, entry, 0)
        np.testing.assert_array_equal(d, h)
        assert all(ds[k] == hs[k] for k in hs)
        assert pieces == 1 or ds["repairs"] > 0


def test_a_long_chain_is_not_a_launch_per_level(lib_built):
    n = 200_000
    x, cand = chain(n, n)
    build(x[:100], cand[:100] % 100, 0, 0)
    best = 1e9
    for _ in range(3):
        t = time.perf_counter()
        build(x, cand, 0, 0)
        best = min(best, time.perf_counter() - t)
    assert best < 0.25  # 15 ms; 200,000 launches take 1.2 s, and cannot take less than 0.3
