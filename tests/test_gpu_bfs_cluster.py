"""GPU parity of the single-source BFS where it starts in the thread-block cluster: graphs
whose rows are short (the search can be handed over to the whole grid) and graphs small
enough to be searched there whole.  Depths equal the oracle's, parents are valid."""
import numpy as np
import pytest

import oracle
import synth
from checks import assert_valid_parents
from paper_1804_03327_gb300 import gbx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def tree(fanout, n):
    """Complete tree: its levels grow by the fanout, so the frontier outgrows the cluster
    (24,576 vertices) and, for wide ones, a block's queue (8,192) within one level."""
    d = np.arange(1, n, dtype=np.int32)
    return n, ((d - 1) // fanout).astype(np.int32), d


def ring(n, k):
    """Every vertex joined to the k next ones: rows of 2k entries, around the five that the
    dense arrays hold and the 32 that make a mesh."""
    s = np.repeat(np.arange(n, dtype=np.int32), k)
    d = (s + np.tile(np.arange(1, k + 1, dtype=np.int32), n)) % n
    return n, s, d.astype(np.int32)


def grid(w, h, p=0.01):
    n, s, d = synth.grid_edges(w, h, p_delete=p, seed=w)
    return n, s, d


def rmat(scale, ef):
    return synth.rmat_edges(scale, ef, seed=scale)


CASES = {
    "grid-1x1": (lambda: grid(1, 1), True),
    "grid-1x9": (lambda: grid(1, 9, 0.0), True),
    "grid-333x211": (lambda: grid(333, 211), True),  # above 65,536 vertices: outputs filled by the grid
    "grid-251x261": (lambda: grid(251, 261), True),
    "tree2": (lambda: tree(2, 150001), True),
    "tree20": (lambda: tree(20, 170001), True),
    "tree31-directed": (lambda: tree(31, 1000003), False),
    "ring1": (lambda: ring(3001, 1), True),
    "ring2-directed": (lambda: ring(70001, 2), False),
    "ring3": (lambda: ring(9001, 3), True),
    "ring16": (lambda: ring(40001, 16), True),
    "ring17": (lambda: ring(40001, 17), True),  # rows of 34: not a mesh
    "rmat10": (lambda: rmat(10, 16), True),
    "rmat13-directed": (lambda: rmat(13, 8), False),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_cluster_bfs(name):
    make, sym = CASES[name]
    n, s, d = make()
    s, d = np.ascontiguousarray(s, np.int32), np.ascontiguousarray(d, np.int32)
    og = oracle.graph(n, s, d, symmetrize=sym)
    g = gbx.graph_build(n, s, d, symmetrize=sym)
    want = {}
    for src in {0, n // 2, n - 1}:
        for direction in (gbx.DIR_AUTO, gbx.DIR_PUSH):
            # one buffer on a 16-byte boundary, one off it
            depth = torch.full((n + 1,), 9, dtype=torch.int32, device="cuda")[1:]
            parent = torch.full((n,), 9, dtype=torch.int32, device="cuda")
            for _ in range(2):  # again on the same scratch
                gbx.bfs(g, src, depth, parent, gbx.desc_init(direction=direction))
            gbx.graph_sync(g)
            if src not in want:
                want[src] = oracle.bfs(og, src)[0]
            got = depth.cpu().numpy()
            assert np.array_equal(got, want[src]), (src, direction)
            if n <= 100000:
                assert_valid_parents(og.out_ptr, og.out_col, got, parent.cpu().numpy(), src)
    # a traced run follows Section 6.3's rule on the whole grid: the same depths
    depth = torch.empty(n, dtype=torch.int32, device="cuda")
    gbx.bfs(g, 0, depth, None, gbx.desc_init(trace=1))
    gbx.graph_sync(g)
    assert np.array_equal(depth.cpu().numpy(), want[0])
    g.free()


@pytest.mark.parametrize("blocks", [0, 1, 2])
@pytest.mark.parametrize("scale,ef", [(14, 16), (19, 12), (20, 16)])
def test_grid_size(scale, ef, blocks):
    """The whole grid with one and with two blocks per SM, on both sides of the size where the default changes."""
    n, s, d = rmat(scale, ef)
    og, g = oracle.graph(n, s, d), gbx.graph_build(n, s, d)
    src = int(s[0])
    want, _, _ = oracle.bfs(og, src)
    depth = torch.empty(n, dtype=torch.int32, device="cuda")
    parent = torch.empty(n, dtype=torch.int32, device="cuda")
    gbx.bfs(g, src, depth, parent, gbx.desc_init(blocks_per_sm=blocks))
    gbx.graph_sync(g)
    assert np.array_equal(depth.cpu().numpy(), want)
    assert_valid_parents(og.out_ptr, og.out_col, want, parent.cpu().numpy(), src)
