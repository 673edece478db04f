"""The CUDA-core rotation's three tile sizes (8 x 32, 32 x 64, 64 x 128 queries
x outputs, chosen by the number of tiles) at their edges, bit for bit against
the chunked fp32 order written out: 32-column fmaf chains, sums in order."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("d", [32, 96, 128, 160, 288])
@pytest.mark.parametrize("nq", [1, 7, 8, 9, 63, 65, 700, 2433, 40_001])
def test_rotation_tiles(tmp_path, lib_built, d, nq):
    from paper_2411_12229_gb300 import index_builder as ib
    from paper_2411_12229_gb300.api import Index
    g = np.random.default_rng(d)
    p = tmp_path / "r.sqg"
    ib.build_index(p, g.standard_normal((100, d)).astype(np.float32), 32)
    rot = torch.from_numpy(ib.random_rotation(d, 2)).cuda().double()
    q = torch.randn((nq, d), generator=torch.Generator(device="cuda").manual_seed(nq), device="cuda")
    got = Index(p, 0).prepare_queries(q)[0]
    rows = torch.unique(torch.cat([torch.arange(min(nq, 80)), torch.arange(max(0, nq - 80), nq)])).cuda()
    x = q[rows].double()
    total = torch.zeros((len(rows), d), dtype=torch.float32, device="cuda")
    for c in range(0, d, 32):
        acc = torch.zeros_like(total)
        for j in range(c, c + 32):
            # a product of two fp32 numbers is exact in fp64; adding the fp32
            # accumulator there and rounding is an fma unless the fp64 sum was
            # itself rounded, which the comparison below allows for
            acc = (x[:, j:j + 1] * rot[:, j][None, :] + acc.double()).float()
        total = total + acc
    same = got[rows] == total
    # double rounding happens about once in 2^29 sums; a wrong order or tile
    # changes a large share of the values
    assert float((~same).float().mean()) <= 1e-5
