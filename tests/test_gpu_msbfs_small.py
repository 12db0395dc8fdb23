"""GPU parity of batches on small graphs, where they are cut differently from large ones: the output
rows are written by as many warps as there are, in pieces of 32 vertices and a few rows."""
import numpy as np
import pytest

import oracle
import synth
from paper_1804_03327_gb300 import gbx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def check(n, s, d, sym, S, descs, dtype=torch.int16, distinct=24, shift=0, seed=1):
    og, g = oracle.graph(n, s, d, symmetrize=sym), gbx.graph_build(n, s, d, symmetrize=sym)
    r = np.random.default_rng(seed)
    pool = r.integers(0, n, distinct).astype(np.int32)
    srcs = pool[r.integers(0, distinct, S)]
    want = {int(v): oracle.bfs(og, int(v))[0] for v in pool}
    want = np.stack([want[int(v)] for v in srcs])
    for desc in descs:
        flat = torch.full((S * n + shift,), 77, dtype=dtype, device="cuda")
        depth = flat[shift:].view(S, n)  # rows on and off the boundaries of wide stores
        gbx.bfs_batch(g, srcs, depth, desc)
        gbx.graph_sync(g)
        got = depth.cpu().numpy().astype(np.int32)
        assert np.array_equal(got, want), np.argwhere(got != want)[:3]
        assert torch.all(flat[:shift] == 77)
    g.free()


@pytest.mark.parametrize("n", [1, 2, 31, 33, 127, 129, 500, 4097])
@pytest.mark.parametrize("S", [1, 5, 32, 33, 64, 65, 130, 300])
def test_output_rows(n, S):
    """A path through a third of the vertices (depths beyond 16, stored when found) beside random edges."""
    r = np.random.default_rng(n)
    p = np.arange(max(1, n // 3), dtype=np.int32)
    e = r.integers(n // 3, n, (2, n)).astype(np.int32) if n > 2 else np.zeros((2, 1), np.int32)
    s, d = np.concatenate([p[:-1], e[0]]), np.concatenate([p[1:], e[1]])
    for dtype, shift in ((torch.int16, 0), (torch.int16, 3), (torch.int32, 0), (torch.int32, 1)):
        check(n, s, d, True, S, [gbx.desc_init()], dtype, distinct=8, shift=shift, seed=S)


@pytest.mark.parametrize("alpha", [0.0, 1e-9, 0.01, 0.25, 0.5, 0.999, 1.0, 1e30, float("inf")])
def test_direction_is_the_edge_quotient(alpha):
    """AUTO pulls once the active edges exceed alpha * nnz, the product in binary64."""
    n, s, d = synth.rmat_edges(9, 8, seed=5)
    og, g = oracle.graph(n, s, d), gbx.graph_build(n, s, d)
    srcs = synth.sources(n, s, d, 7, seed=2).astype(np.int32)
    depth = torch.empty((7, n), dtype=torch.int32, device="cuda")
    gbx.bfs_batch(g, srcs, depth, gbx.desc_init(alpha=alpha))
    gbx.graph_sync(g)
    for b, v in enumerate(srcs):
        assert np.array_equal(depth[b].cpu().numpy(), oracle.bfs(og, int(v))[0])
    tr = gbx.bfs_batch_trace(g)
    pull = tr["mf"].astype(np.float64) > np.float64(np.float32(alpha)) * np.float64(og.nnz)
    assert np.array_equal(tr["direction"] == gbx.DIR_PULL, pull)
    # alpha a quotient of binary32 that a level meets exactly
    for mf in set(int(x) for x in tr["mf"]):
        for a in (np.float32(mf / og.nnz), np.nextafter(np.float32(mf / og.nnz), np.float32(0))):
            gbx.bfs_batch(g, srcs, depth, gbx.desc_init(alpha=float(a)))
            gbx.graph_sync(g)
            t = gbx.bfs_batch_trace(g)
            assert np.array_equal(t["direction"] == gbx.DIR_PULL,
                                  t["mf"].astype(np.float64) > np.float64(a) * np.float64(og.nnz))
    g.free()


def hubs(n, directed, seed):
    """Random edges with some rows of in-degree around the five dense entries, the lane's share and the
    24 more it takes, a few hundred, and thousands (beyond the warp's 2,048); directed: sinks too."""
    r = np.random.default_rng(seed)
    s, d = [r.integers(0, n // 2, 2 * n)], [r.integers(0, n, 2 * n)]
    for k, deg in enumerate([4, 5, 6, 12, 13, 14, 36, 37, 38, 40, 300, 700, 2060, 2100, min(n - 1, 9000), n // 2]):
        deg = min(deg, n // 2)
        d.append(np.full(deg, (n - 1 - 7 * k) % n if k % 2 else (3 + 5 * k) % n))
        s.append(r.permutation(n // 2)[:deg])
    return n, np.concatenate(s).astype(np.int32), np.concatenate(d).astype(np.int32), not directed


@pytest.mark.parametrize("n", [97, 3000, 20011, 50021, 160001])
@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("S", [1, 20, 64])
def test_one_word(n, directed, S):
    n, s, d, sym = hubs(n, directed, n)
    descs = [gbx.desc_init(), gbx.desc_init(direction=gbx.DIR_PULL), gbx.desc_init(alpha=0.2, pull_probe=4),
             gbx.desc_init(direction=gbx.DIR_PULL, pull_probe=100), gbx.desc_init(blocks_per_sm=3)]
    check(n, s, d, sym, S, descs, distinct=min(S, 12))


@pytest.mark.parametrize("S", [20, 64, 100, 200, 300, 700, 2100, 4100])
@pytest.mark.parametrize("n,directed", [(3, False), (90, True), (2999, True), (9001, False), (19001, True),
                                        (40009, False), (90001, True)])
def test_teams(n, directed, S):
    """Teams of 4 to 32 lanes a row and none (too many vertices for the words), one to 66 words."""
    if n * S > 40_000_000:
        pytest.skip("the same forms as with fewer sources")
    n, s, d, sym = hubs(n, directed, n + S)
    descs = [gbx.desc_init(), gbx.desc_init(direction=gbx.DIR_PULL), gbx.desc_init(alpha=0.1, blocks_per_sm=3)]
    check(n, s, d, sym, S, descs, distinct=min(S, 10))


@pytest.mark.parametrize("S", [3, 130])
@pytest.mark.parametrize("n,deg", [(6000, 2400), (4000, 600)])
def test_long_rows_only(n, deg, S):
    """Every row is long: more in a block than it takes together (32), and none for the lanes alone."""
    v = np.arange(n, dtype=np.int64)
    s = ((v[:, None] + 1 + np.arange(deg)) % n).reshape(-1).astype(np.int32)
    d = np.repeat(v, deg).astype(np.int32)
    check(n, s, d, False, S, [gbx.desc_init(direction=gbx.DIR_PULL), gbx.desc_init()], distinct=3)
