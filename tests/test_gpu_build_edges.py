"""GPU parity of the graph build and the weights at the edges of their tiles: edge counts
around the sort's 4,096 and the deduplication's 2,048 keys, vertex counts at powers of two
(where the key of a dropped self-loop is all ones), rows from empty to thousands of entries,
names that are anything but spread evenly.  CSR and weights equal the oracle's exactly."""
import numpy as np
import pytest

import oracle
from paper_1804_03327_gb300 import gbx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def edges(n, m, kind, rng):
    if kind == "uniform":
        return rng.integers(0, n, m), rng.integers(0, n, m)
    if kind == "loops":  # most entries are dropped, some at the very last vertex
        s = np.where(rng.random(m) < 0.5, n - 1, rng.integers(0, n, m))
        return s, np.where(rng.random(m) < 0.8, s, rng.integers(0, n, m))
    if kind == "hub":  # one row of thousands, its neighbours bunched at one end
        return np.zeros(m, np.int64), (n - 1) - np.minimum(rng.geometric(0.01, m), n - 1)
    return np.full(m, n // 2), np.full(m, n - 1)  # one pair again and again


@pytest.mark.parametrize("n", [1, 2, 31, 64, 1000, 4096, 65537])
@pytest.mark.parametrize("m", [0, 1, 2047, 2048, 2049, 4095, 4097, 30000])
@pytest.mark.parametrize("kind", ["uniform", "loops", "hub", "same"])
def test_build_and_weights(n, m, kind):
    rng = np.random.default_rng(n + m)
    s, d = (np.ascontiguousarray(x, np.int32) for x in edges(n, m, kind, rng))
    w = rng.random(m).astype(np.float32) - np.float32(0.2)
    for sym in (True, False):
        for drop in (True, False):
            if drop:
                og = oracle.graph_weighted(n, s, d, w, symmetrize=sym)
            else:
                og = oracle.graph(n, s, d, symmetrize=sym, drop_self_loops=False)
            g = gbx.graph_build(n, torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda(), symmetrize=sym,
                                drop_self_loops=drop)
            for t, (op, oc) in enumerate([(og.out_ptr, og.out_col), (og.in_ptr, og.in_col)]):
                rp, col = gbx.graph_copy_csr(g, bool(t))
                assert np.array_equal(rp, op) and np.array_equal(col, oc), (sym, drop, t)
            if drop and m > 0:
                gbx.graph_set_weights(g, s, d, w)
                assert np.array_equal(gbx.graph_weights(g, False), og.out_val)
                assert np.array_equal(gbx.graph_weights(g, True), og.in_val)
            g.free()


def test_a_build_that_found_no_memory_leaves_the_next_one_alone():
    n, s, d = 30_000_000, np.zeros(1, np.int32), np.ones(1, np.int32)  # some 2.5 GB
    gbx.graph_build(10, s, d).free()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    held = torch.empty(free - (300 << 20), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(gbx.GbxError):
            gbx.graph_build(n, s, d)
        g = gbx.graph_build(10, s, d)
        depth = torch.empty(10, dtype=torch.int32, device="cuda")
        gbx.bfs(g, 0, depth)
        gbx.graph_sync(g)
        assert depth.tolist() == [0, 1] + [-1] * 8
        g.free()
    finally:  # the memory goes back to the device, not only to the allocator's cache
        del held
        torch.cuda.empty_cache()
