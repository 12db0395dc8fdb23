"""GPU parity of gbx_sssp where it runs in the thread-block cluster (short rows, non-negative
weights): distances equal the oracle's binary32 ones bit for bit, whatever the order of
relaxations, also where the search is handed over to the whole grid."""
import numpy as np
import pytest

import oracle
import synth
from paper_1804_03327_gb300 import gbx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def ring(n, k):
    s = np.repeat(np.arange(n, dtype=np.int32), k)
    d = (s + np.tile(np.arange(1, k + 1, dtype=np.int32), n)) % n
    return n, s, d.astype(np.int32)


def scattered(n, k, seed):
    """k random out-edges a vertex, rows of at most 32: the frontier explodes, so the grid takes over."""
    rng = np.random.default_rng(seed)
    return n, np.repeat(np.arange(n, dtype=np.int32), k), rng.integers(0, n, n * k).astype(np.int32)


GRAPHS = {
    "grid-1x1": (lambda: synth.grid_edges(1, 1, p_delete=0.0, seed=1), True),
    "grid-2x5": (lambda: synth.grid_edges(2, 5, p_delete=0.0, seed=1), True),
    "grid-90x71": (lambda: synth.grid_edges(90, 71, p_delete=0.02, seed=2), True),
    "grid-401x203": (lambda: synth.grid_edges(401, 203, p_delete=0.01, seed=3), True),
    "ring2-directed": (lambda: ring(5003, 2), False),
    "ring3": (lambda: ring(2001, 3), True),
    "ring16": (lambda: ring(3001, 16), True),  # rows of 32: the longest a mesh has
    "scattered-directed": (lambda: scattered(200003, 4, 5), False),
}
WEIGHTS = {
    "real": lambda r, m: r.random(m).astype(np.float32) * 0.9 + np.float32(0.1),
    "integer": lambda r, m: r.integers(1, 65, m).astype(np.float32),
    "zero": lambda r, m: np.zeros(m, np.float32),
    "spread": lambda r, m: np.exp(r.uniform(-40, 40, m)).astype(np.float32),  # 34 decades
    "some-zero": lambda r, m: (r.random(m) < 0.5).astype(np.float32),
    "negative": lambda r, m: -np.zeros(m, np.float32),  # -0.0 is not negative
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
@pytest.mark.parametrize("weights", sorted(WEIGHTS))
def test_cluster_sssp(name, weights):
    make, sym = GRAPHS[name]
    n, s, d = make()
    s, d = np.ascontiguousarray(s, np.int32), np.ascontiguousarray(d, np.int32)
    w = WEIGHTS[weights](np.random.default_rng(7), len(s))
    og = oracle.graph_weighted(n, s, d, w, symmetrize=sym)
    g = gbx.graph_build(n, s, d, symmetrize=sym)
    gbx.graph_set_weights(g, s, d, w)
    for src in {0, n // 2}:
        want = oracle.sssp(og, src)[0]
        for direction in (gbx.DIR_AUTO, gbx.DIR_PUSH):
            dist = torch.full((n,), -1.0, dtype=torch.float32, device="cuda")
            gbx.sssp(g, src, dist, gbx.desc_init(direction=direction))
            gbx.graph_sync(g)
            assert np.array_equal(dist.cpu().numpy(), want), (src, direction)
    # the traced run iterates on the whole grid: the same distances
    gbx.sssp(g, 0, dist, gbx.desc_init(trace=1))
    gbx.graph_sync(g)
    assert np.array_equal(dist.cpu().numpy(), oracle.sssp(og, 0)[0])
    g.free()


def test_weights_replaced_by_negative_ones():
    """A weight below zero takes the search back to the grid's iterations."""
    n, s, d = ring(4001, 2)
    g = gbx.graph_build(n, s, d, symmetrize=False)
    rng = np.random.default_rng(3)
    for low in (0.5, -0.1):
        w = rng.uniform(0.5, 2.0, len(s)).astype(np.float32)
        w[::2] = np.where(rng.random(len(w[::2])) < 0.01, np.float32(low), w[::2])
        gbx.graph_set_weights(g, s, d, w)
        dist = torch.empty(n, dtype=torch.float32, device="cuda")
        gbx.sssp(g, 1, dist)
        gbx.graph_sync(g)
        want = oracle.sssp(oracle.graph_weighted(n, s, d, w, symmetrize=False), 1)[0]
        if low > 0:
            assert np.array_equal(dist.cpu().numpy(), want)
        else:  # with negative weights the rounding depends on the schedule
            assert np.allclose(dist.cpu().numpy(), want, rtol=1e-4)
    g.free()


def test_weights_without_memory_for_the_mesh_records():
    """The records only make searches faster: weights are accepted where there is no room for them."""
    n = 8_000_000  # weights and row list: 128 MB, the records: 256 MB
    s = torch.arange(n - 1, dtype=torch.int32, device="cuda")
    w = torch.ones(n - 1, dtype=torch.float32, device="cuda")
    small = gbx.graph_build(3, s[:2].contiguous(), (s[:2] + 1).contiguous())
    gbx.graph_set_weights(small, s[:2].contiguous(), (s[:2] + 1).contiguous(), w[:2].contiguous())  # kernels loaded
    # a path of 1,000 vertices among pairs, so that the whole grid has few iterations
    d = torch.where((s < 1000) | (s % 2 == 0), s + 1, s)
    g = gbx.graph_build(n, s, d)
    dist = torch.empty(n, dtype=torch.float32, device="cuda")
    want = np.full(n, np.inf, np.float32)
    want[:1002] = np.arange(1002)
    gbx.sssp(small, 0, torch.empty(3, dtype=torch.float32, device="cuda"))
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    held = torch.empty(free - (200 << 20), dtype=torch.uint8, device="cuda")
    try:
        for room in (False, True):
            if room:
                held = None
                torch.cuda.empty_cache()
            gbx.graph_set_weights(g, s, d, w)
            dist.fill_(-1.0)
            gbx.sssp(g, 0, dist)
            gbx.graph_sync(g)
            assert np.array_equal(dist.cpu().numpy(), want)
    finally:  # the memory goes back to the device, not only to the allocator's cache
        held = None
        torch.cuda.empty_cache()
    g.free()
    small.free()
