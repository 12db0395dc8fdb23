"""GPU parity of the batched BFS where its lane-word groups can go wrong: every group
width (W = 1, 2, 4, 8, 12, 36 words and, above 64 words, two chunks), ragged last words,
rows long enough to be deferred to the whole grid (in-degrees of about 5,700 and 7,800),
directed graphs with vertices nobody leaves, odd vertex counts (output rows that no
vector store fits) and depths on both sides of 16.  Depths equal the oracle's exactly."""
import numpy as np
import pytest

import oracle
import synth
from paper_1804_03327_gb300 import gbx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

_cache = {}


def graph(name):
    if name not in _cache:
        if name == "chain":  # a path with a dense end: depths 0 .. 40 in one batch
            k = 40
            a, b = np.triu_indices(30, 1)
            s = np.concatenate([np.arange(k), k + a]).astype(np.int32)
            d = np.concatenate([np.arange(1, k + 1), k + b]).astype(np.int32)
            n, directed = k + 30 + 3, False
        else:
            directed = name == "hubs-directed"
            n, s, d = synth.rmat_edges(13, 8, seed=21)
            hs, hd = [s], [d]
            for h, p in ((0, 0.7), (1, 0.95)):
                v = np.flatnonzero(synth.vertex_set(n, p, seed=6, stream=h + 1)).astype(np.int32)
                hs.append(v if directed else np.full(len(v), h, np.int32))
                hd.append(np.full(len(v), h, np.int32) if directed else v)
            s, d, n = np.concatenate(hs), np.concatenate(hd), n + 3
        _cache[name] = (n, s, d, oracle.graph(n, s, d, symmetrize=not directed),
                        gbx.graph_build(n, s, d, symmetrize=not directed))
    return _cache[name]


@pytest.mark.parametrize("name", ["hubs", "hubs-directed", "chain"])
@pytest.mark.parametrize("S", [3, 64, 66, 130, 500, 700, 2100, 4200])
@pytest.mark.parametrize("direction", [gbx.DIR_AUTO, gbx.DIR_PUSH, gbx.DIR_PULL])
def test_lane_groups(name, S, direction):
    n, s, d, og, g = graph(name)
    pool = synth.sources(n, s, d, 64, seed=S)
    srcs = pool[np.arange(S) % len(pool)]  # repeated sources: the oracle runs each once
    dtype = torch.int16 if S % 4 else torch.int32
    depth = torch.full((S, n), 77, dtype=dtype, device="cuda")
    gbx.bfs_batch(g, srcs, depth, gbx.desc_init(direction=direction))
    gbx.graph_sync(g)
    want = {int(v): oracle.bfs(og, int(v))[0] for v in pool[: min(S, len(pool))]}
    got = depth.cpu().numpy().astype(np.int32)
    for b, v in enumerate(srcs):
        assert np.array_equal(got[b], want[int(v)]), (b, int(v))


@pytest.mark.parametrize("w,h", [(1, 1), (3, 1), (1, 700), (37, 41), (300, 211)])
@pytest.mark.parametrize("S", [1, 31, 64])
@pytest.mark.parametrize("k", [0, 3, 16])
def test_mesh_batches(w, h, S, k):
    """One lane word on graphs of short rows (the push without a degree prefix): grids, and
    rings joined to the k next vertices (rows of 2k entries: beyond the five of the dense
    arrays, up to the 32 that make a mesh), in every direction, int16 and int32 rows."""
    n, s, d = synth.grid_edges(w, h, p_delete=0.02, seed=h)
    if k:
        n = min(w * h, 2500) + 40
        s = np.repeat(np.arange(n, dtype=np.int32), k)
        d = ((s + np.tile(np.arange(1, k + 1, dtype=np.int32), n)) % n).astype(np.int32)
    og, g = oracle.graph(n, s, d), gbx.graph_build(n, s, d)
    srcs = (np.arange(S) * 7919 % n).astype(np.int32)
    want = {int(v): oracle.bfs(og, int(v))[0] for v in set(srcs[:16])}
    for direction, alpha in ((gbx.DIR_AUTO, 1e30), (gbx.DIR_AUTO, 0.01), (gbx.DIR_PUSH, 0.0), (gbx.DIR_PULL, 0.0)):
        for dtype in (torch.int16, torch.int32):
            depth = torch.full((S, n), 55, dtype=dtype, device="cuda")
            gbx.bfs_batch(g, srcs, depth, gbx.desc_init(direction=direction, alpha=alpha))
            gbx.graph_sync(g)
            tr = gbx.bfs_batch_trace(g)
            got = depth.cpu().numpy().astype(np.int32)
            for b in range(min(S, 16)):
                assert np.array_equal(got[b], want[int(srcs[b])]), (direction, b)
            assert tr["n_new"].sum() == np.sum(got > 0) and np.all(tr["mf"][1:] == tr["mf_new"][:-1])
            # the active vertices of a level, each once however often it was listed
            deg = np.diff(og.out_ptr)
            active = [(got == level).any(axis=0) & (deg > 0) for level in range(len(tr))]
            assert [int(x) for x in tr["nf"]] == [int(x.sum()) for x in active]
            assert [int(x) for x in tr["mf"]] == [int(deg[x].sum()) for x in active]
    g.free()


@pytest.mark.parametrize("k", [1, 2, 5, 12])
@pytest.mark.parametrize("dtype", [torch.int16, torch.int32])
def test_lists_beyond_the_queue_arrays(k, dtype):
    """Disjoint complete graphs of five vertices, every vertex a source: nnz = 4 n, and every edge lists its
    end at the first level, 4 n entries where the queue arrays hold 3 n."""
    a, b = np.triu_indices(5, 1)
    n = 5 * k
    s = (np.arange(k)[:, None] * 5 + a).reshape(-1).astype(np.int32)
    d = (np.arange(k)[:, None] * 5 + b).reshape(-1).astype(np.int32)
    g = gbx.graph_build(n, s, d)
    assert g.info()[1] == 4 * n
    depth = torch.full((n, n), 55, dtype=dtype, device="cuda")
    v = np.arange(n)
    want = np.where(v[:, None] // 5 == v // 5, 1, -1) + np.where(v[:, None] == v, -1, 0)
    for _ in range(3):
        gbx.bfs_batch(g, v.astype(np.int32), depth, gbx.desc_init(alpha=1e30))
        gbx.graph_sync(g)
        assert np.array_equal(depth.cpu().numpy(), want)
        tr = gbx.bfs_batch_trace(g)
        assert [int(x) for x in tr["nf"]] == [n, n] and [int(x) for x in tr["n_new"]] == [4 * n, 0]
    g.free()
