"""The clusters' bounded wait, without a fault: a block that withholds its counts lets every block's
wait run out; all of them leave, the host reads GBX_ERR_TIMEOUT once, and the next searches on the
same graph are right."""
import numpy as np
import pytest

import oracle
import synth
from paper_1804_03327_gb300 import gbx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("w,h", [(1, 1), (31, 17), (400, 301)])
def test_cluster_wait_times_out_and_the_graph_stays_usable(w, h):
    n, s, d = synth.grid_edges(w, h, p_delete=0.0, seed=3)
    val = np.random.default_rng(1).random(len(s)).astype(np.float32)
    og = oracle.graph_weighted(n, s, d, val)
    g = gbx.graph_build(n, s, d)
    gbx.graph_set_weights(g, s, d, val)
    depth = torch.empty(n, dtype=torch.int32, device="cuda")
    dist = torch.empty(n, dtype=torch.float32, device="cuda")
    want, want_dist = oracle.bfs(oracle.graph(n, s, d), n // 2)[0], oracle.sssp(og, n // 2)[0]
    for which in (gbx.TUNE_BFS, gbx.TUNE_SSSP, gbx.TUNE_BFS):
        if which == gbx.TUNE_SSSP and len(s) == 0:
            continue  # no edges: no records
        gbx.selftest_cluster_timeout(g, which, 3_000_000)  # 3 ms
        gbx.bfs(g, n // 2, depth)  # sees the pending error and leaves
        gbx.sssp(g, n // 2, dist)
        with pytest.raises(gbx.GbxError) as e:
            gbx.graph_sync(g)
        assert e.value.status == gbx.ERR_TIMEOUT
        gbx.graph_sync(g)  # cleared
        for _ in range(2):
            gbx.bfs(g, n // 2, depth)
            gbx.sssp(g, n // 2, dist)
            gbx.graph_sync(g)
            assert np.array_equal(depth.cpu().numpy(), want)
            assert np.array_equal(dist.cpu().numpy(), want_dist)
    g.free()


def test_cluster_timeout_needs_a_cluster():
    n, s, d = synth.rmat_edges(14, 16, seed=2)
    g = gbx.graph_build(n, s, d)
    for which, status in ((gbx.TUNE_BFS, gbx.ERR_NOT_SUPPORTED), (gbx.TUNE_SSSP, gbx.ERR_NOT_SUPPORTED),
                          (gbx.TUNE_BATCH, gbx.ERR_INVALID_VALUE)):
        with pytest.raises(gbx.GbxError) as e:
            gbx.selftest_cluster_timeout(g, which, 1_000_000)
        assert e.value.status == status
    g.free()
