"""Searches that start in the thread-block cluster and outgrow it: rows of up to 32 entries whose
frontiers explode (random k-out and k-regular graphs, small worlds, wide trees), so that the frontier
is handed over at every level from the second on, with queues that spill.  Depths equal the
oracle's; every parent is one level up over an edge, also across the hand-over."""
import numpy as np
import pytest

import oracle
from checks import assert_valid_parents_large
from paper_1804_03327_gb300 import gbx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def k_out(n, k, seed):
    r = np.random.default_rng(seed)
    return n, np.repeat(np.arange(n, dtype=np.int32), k), r.integers(0, n, n * k).astype(np.int32)


def regular(n, k, seed):
    r = np.random.default_rng(seed)
    p = [r.permutation(n).astype(np.int32) for _ in range(k // 2)]
    return n, np.concatenate(p), np.concatenate([np.roll(q, 1) for q in p])


def world(n, k, seed):
    r = np.random.default_rng(seed)
    s = np.repeat(np.arange(n, dtype=np.int32), k)
    d = (s + np.tile(np.arange(1, k + 1, dtype=np.int32), n)) % n
    far = r.random(n * k) < 0.02
    return n, s, np.where(far, r.integers(0, n, n * k), d).astype(np.int32)


def tree(fanout, n):
    d = np.arange(1, n, dtype=np.int32)
    return n, ((d - 1) // fanout).astype(np.int32), d


CASES = {
    "regular4-30k": (lambda: regular(30001, 4, 1), True),
    "regular16-30k": (lambda: regular(30011, 16, 2), True),
    "regular16-9k": (lambda: regular(9001, 16, 3), True),
    "k-out16-30k": (lambda: k_out(30007, 16, 4), False),
    "k-out32-120k": (lambda: k_out(120011, 32, 5), False),
    "world4-60k": (lambda: world(60013, 4, 6), True),
    "tree2": (lambda: tree(2, 150001), True),
    "tree20": (lambda: tree(20, 170001), True),
    "tree31-directed": (lambda: tree(31, 1000003), False),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_bfs_across_the_handover(name):
    make, sym = CASES[name]
    n, s, d = make()
    og = oracle.graph(n, s, d, symmetrize=sym)
    g = gbx.graph_build(n, s, d, symmetrize=sym)
    pairs = (np.concatenate([s, d]), np.concatenate([d, s])) if sym else (s, d)
    for src in (0, n // 2):
        want = oracle.bfs(og, src)[0]
        for desc in (gbx.desc_init(), gbx.desc_init(direction=gbx.DIR_PUSH), gbx.desc_init(alpha=0.3, beta=0.2)):
            depth = torch.full((n,), 9, dtype=torch.int32, device="cuda")
            parent = torch.full((n,), 9, dtype=torch.int32, device="cuda")
            gbx.bfs(g, src, depth, parent, desc)
            gbx.graph_sync(g)
            got = depth.cpu().numpy()
            assert np.array_equal(got, want), src
            assert_valid_parents_large(n, pairs, got, parent.cpu().numpy(), src)
    g.free()


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("integer", [0, 1])
def test_sssp_across_the_handover(name, integer):
    make, sym = CASES[name]
    n, s, d = make()
    r = np.random.default_rng(11)
    w = (r.integers(1, 65, len(s)) if integer else r.random(len(s)) * 0.9 + 0.1).astype(np.float32)
    og = oracle.graph_weighted(n, s, d, w, symmetrize=sym)
    g = gbx.graph_build(n, s, d, symmetrize=sym)
    gbx.graph_set_weights(g, s, d, w)
    want = oracle.sssp(og, n // 3)[0]
    for direction in (gbx.DIR_AUTO, gbx.DIR_PUSH):
        dist = torch.full((n,), -1.0, dtype=torch.float32, device="cuda")
        gbx.sssp(g, n // 3, dist, gbx.desc_init(direction=direction))
        gbx.graph_sync(g)
        assert np.array_equal(dist.cpu().numpy(), want), direction
    g.free()


@pytest.mark.parametrize("n", [300, 8192, 8193])
@pytest.mark.parametrize("entries", [72 * 1024 - 2, 72 * 1024, 72 * 1024 + 2])
def test_bfs_around_the_size_of_a_whole_search(n, entries):
    r = np.random.default_rng(entries)
    key = np.unique(r.integers(0, n, 200000).astype(np.int64) * n + r.integers(0, n, 200000))
    s, d = key // n, key % n
    keep = r.permutation(np.flatnonzero(s < d))[: entries // 2]
    s, d = s[keep].astype(np.int32), d[keep].astype(np.int32)
    g = gbx.graph_build(n, s, d)
    assert g.info()[1] == min(entries, 2 * len(s))
    og = oracle.graph(n, s, d)
    for src in (int(s[0]), int(d[-1])):
        depth = torch.empty(n, dtype=torch.int32, device="cuda")
        parent = torch.empty(n, dtype=torch.int32, device="cuda")
        gbx.bfs(g, src, depth, parent)
        gbx.graph_sync(g)
        got = depth.cpu().numpy()
        assert np.array_equal(got, oracle.bfs(og, src)[0])
        assert_valid_parents_large(n, (np.concatenate([s, d]), np.concatenate([d, s])), got, parent.cpu().numpy(), src)
    g.free()
