"""A search's plan.  It asks the driver once per kernel build and size: the
plan of a used handle, in any order and from several threads, is that of a
fresh one.  A batch that is resident at once takes larger visited tables only
as far as the warps of other streams' batches still find room."""

import ctypes as C
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


@pytest.mark.parametrize("d,R", [(96, 32), (128, 32), (256, 32), (128, 64), (960, 64), (1536, 32)])
def test_larger_tables_leave_room(tmp_path, lib_built, d, R):
    from paper_2411_12229_gb300 import _binding as B
    from paper_2411_12229_gb300 import index_builder as ib
    from paper_2411_12229_gb300 import synth
    from paper_2411_12229_gb300.api import Index
    p = tmp_path / "i.sqg"
    ib.build_index(p, synth.base(synth.small(synth.BATCHED_1M_D128.with_(d=d), 400, 1)), R)
    ix = Index(p, 0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count

    def plan(nq, k, ef, slots=0, **kw):
        out = (C.c_int32 * 4)()
        params = ix.params(visited_smem_log2=slots, **kw)
        B.check(B.lib().sqg_search_plan(ix.handle, nq, k, ef, C.byref(params), out), "sqg_search_plan")
        return list(out)

    stop = torch.zeros(B.MLP_NPARAM, device="cuda")
    larger = 0
    for k, ef in ((1, 1), (10, 40), (10, 64), (10, 120), (10, 200), (100, 160), (100, 256), (10, 400), (128, 1000)):
        for nq in (1, 200, 719, 8 * sms, 8 * sms + 1, 2001, 3000, 10_000):
            kernel, slots, _, resident = plan(nq, k, ef)  # (the deep kernel's rule is residency alone)
            least = plan(nq, k, ef, 9)
            assert kernel in (1, 2) and slots <= 11 and least[1] <= 9
            assert plan(nq, k, ef, stop_mlp=stop)[1] <= 9
            if slots <= 9:
                assert resident == least[3]
                continue
            larger += 1
            assert nq <= resident * sms
            if kernel == 1:
                assert 4 * resident >= 3 * least[3] if d <= 256 else resident == least[3]
                assert slots == 10 or resident == plan(nq, k, ef, 10)[3]
    assert larger > 0
