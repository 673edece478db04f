"""A search's plan asks the driver once per kernel build and size: the plan
of a used handle, in any order and from several threads, is that of a fresh
one."""

import threading

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPES = [(nq, k, ef, kw) for nq in (1, 700, 1216, 1217, 5000, 60_000)
          for k, ef in ((1, 1), (10, 64), (10, 100), (10, 200), (100, 200), (10, 400), (128, 1000), (256, 2048))
          for kw in ({"lean": 0}, {"kernel": 1}, {"lean": 1}, {"visited_smem_log2": 7}, {"warps_per_block": 3},
                     {"team": 16}, {"rotation": 2})]


def test_plans_of_a_used_handle(tiny_index):
    from paper_2411_12229_gb300.api import Index
    path = tiny_index[0]

    def sizes(ix, shapes):
        return {i: ix.workspace_size(nq, k, ef, **kw) for i, (nq, k, ef, kw) in shapes}

    every = list(enumerate(SHAPES))
    fresh = {}
    for i, shape in every:
        ix = Index(path, 0)
        fresh.update(sizes(ix, [(i, shape)]))
        ix.close()
    ix, got = Index(path, 0), [None] * 4

    def work(t):
        order = every[t::4] + every[::-1] + every
        got[t] = sizes(ix, order)

    ts = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert got == [fresh] * 4
