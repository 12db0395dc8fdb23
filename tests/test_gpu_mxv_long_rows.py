"""The matvec's pull where one block has many rows of thousands of entries: more than its list
holds, each with its only hit (if any) anywhere in the row, with and without early exit."""
import numpy as np
import pytest

import oracle
from paper_1804_03327_gb300 import gbx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("early_exit", [0, 1])
@pytest.mark.parametrize("ones", [0, 1, 40, 10000])
def test_many_long_rows_of_one_block(ones, early_exit):
    n, hubs = 20000, 100  # vertices 0 .. 99 are one block's
    rng = np.random.default_rng(ones)
    lengths = rng.integers(1100, 9000, hubs)
    d = np.repeat(np.arange(hubs, dtype=np.int32), lengths)
    s = rng.integers(hubs, n, len(d)).astype(np.int32)
    u_h = np.zeros(n, np.uint8)
    u_h[rng.integers(hubs, n, ones)] = 1
    og = oracle.graph(n, s, d, symmetrize=False)
    want = oracle.mxv(n, n, og.out_ptr, og.out_col, u_h, None, transpose=True)
    g = gbx.graph_build(n, s, d, symmetrize=False)
    u = torch.from_numpy(u_h).cuda()
    for _ in range(3):
        w = torch.full((n,), 9, dtype=torch.uint8, device="cuda")
        gbx.mxv(gbx.dense(w), None, gbx.LOR_LAND, g, gbx.dense(u),
                gbx.desc_init(direction=gbx.DIR_PULL, early_exit=early_exit))
        torch.cuda.synchronize()
        assert np.array_equal(w.cpu().numpy(), want)
    g.free()
