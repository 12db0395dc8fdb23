"""Pulls of gbx_mxv over graphs whose tiles are several words wide (a warp's words are spread over the
bitmap): row counts around the tile counts, masks that leave one contiguous band of rows."""
import numpy as np
import pytest

import oracle
import synth
from paper_1804_03327_gb300 import gbx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("early_exit", [1, 0])
@pytest.mark.parametrize("width,height", [(1, 1), (33, 1), (557, 559), (1001, 777), (1500, 1399)])
def test_pull_tiles(width, height, early_exit):
    n, s, d = synth.grid_edges(width, height, p_delete=0.01, seed=3)
    og, g = oracle.graph(n, s, d), gbx.graph_build(n, s, d)
    u = synth.vertex_set(n, 0.05, seed=8)
    for lo, hi in [(0, n), (n // 3, n // 3 + max(1, n // 11)), (n - 1, n)]:
        m = np.ones(n, np.uint8)
        m[lo:hi] = 0  # complemented: these rows pass
        want = oracle.mxv(n, n, og.out_ptr, og.out_col, u, m, transpose=True, complement=True)
        ut, mt = torch.from_numpy(u).cuda(), torch.from_numpy(m).cuda()
        w = torch.zeros(n, dtype=torch.uint8, device="cuda")
        gbx.mxv(gbx.dense(w), gbx.dense(mt), gbx.LOR_LAND, g, gbx.dense(ut),
                gbx.desc_init(direction=gbx.DIR_PULL, mask_complement=1, early_exit=early_exit))
        torch.cuda.synchronize()
        assert np.array_equal(w.cpu().numpy(), want), (lo, hi)
