"""The GPU adjust step (batched distances, reverse lists and reachability
flood on the device, rows written by the kernel) against the host's, at the
edges: lists of 1, 4/5, 8/9, 16/17, 32/33 and 512 candidates, d of one chunk,
part of one and several, fewer vertices than R, rows left to the random fill,
vertices that the entry point does not reach, duplicate vectors."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def both(x, cand, R, entry=0, regular=True):
    from paper_2411_12229_gb300 import index_builder as ib
    h, hs = ib.build_graph(x, cand, R, entry, 7, 0, None, regular)
    g, gs = ib.build_graph(x, cand, R, entry, 7, 0, 0, regular)
    np.testing.assert_array_equal(g, h)
    assert all(gs[k] == hs[k] for k in ("avg_nsg_degree", "supplemented", "random_filled", "repairs"))
    return gs


@pytest.mark.parametrize("n,d,R,L", [(200, 32, 32, 1), (200, 96, 32, 4), (300, 128, 32, 5), (300, 160, 32, 8),
                                     (300, 128, 32, 9), (300, 64, 64, 16), (300, 128, 32, 17), (400, 256, 32, 32),
                                     (400, 128, 64, 33), (700, 128, 32, 512), (20, 128, 32, 19), (50, 64, 64, 40),
                                     (2, 32, 32, 1), (260, 544, 32, 70)])
@pytest.mark.parametrize("regular", [True, False])
def test_lists_and_shapes(lib_built, n, d, R, L, regular):
    g = np.random.default_rng(n + d + L)
    x = g.standard_normal((n, d)).astype(np.float32)
    cand = g.integers(0, n, (n, L)).astype(np.uint32)
    cand[g.random((n, L)) < 0.05] = 0xFFFFFFFF
    both(x, cand, R, entry=n // 2, regular=regular)


@pytest.mark.parametrize("regular", [True, False])
def test_unreachable_vertices(lib_built, regular):
    """Clusters whose candidates stay within the cluster: without the random
    fill of regular rows whole clusters have to be connected by the repair,
    over several floods."""
    g = np.random.default_rng(5)
    k, m = 30, 40
    x = (np.repeat(10 * g.standard_normal((k, 64)), m, axis=0) + g.standard_normal((k * m, 64))).astype(np.float32)
    cand = (np.repeat(np.arange(k) * m, m)[:, None] + g.integers(0, m, (k * m, 35))).astype(np.uint32)
    repairs = both(x, cand, 32, entry=3, regular=regular)["repairs"]
    assert regular or repairs > 0


def test_duplicate_vectors(lib_built):
    g = np.random.default_rng(9)
    x = np.repeat(g.standard_normal((60, 128)).astype(np.float32), 5, axis=0)
    both(x, g.integers(0, 300, (300, 90)).astype(np.uint32), 32)


def test_refuses_what_is_not_finite(lib_built):
    from paper_2411_12229_gb300 import _binding as B
    x = np.zeros((100, 32), np.float32)
    x[57, 3] = np.inf
    with pytest.raises(B.SqgError):
        _device_build(x)


def _device_build(x):
    from paper_2411_12229_gb300 import index_builder as ib
    return ib.build_graph(x, np.zeros((100, 8), np.uint32), 32, 0, device=0)
