"""The BFS cluster on graphs whose visited bitmap does not fit its shared memory (more than 7.86M
vertices): a grid walked to the end, and a tree handed over.  Depths in closed form, parents
checked against the shape."""
import numpy as np
import pytest

from paper_1804_03327_gb300 import gbx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def run(g, n, src, desc):
    depth = torch.full((n,), 9, dtype=torch.int32, device="cuda")
    parent = torch.full((n,), 9, dtype=torch.int32, device="cuda")
    gbx.bfs(g, src, depth, parent, desc)
    gbx.graph_sync(g)
    return depth, parent


@pytest.mark.parametrize("w,h", [(2900, 2801), (40, 196700)])
def test_grid(w, h):
    n = w * h
    v = torch.arange(n, dtype=torch.int32, device="cuda").view(h, w)
    s = torch.cat([v[:, :-1].reshape(-1), v[:-1].reshape(-1)])
    d = torch.cat([v[:, 1:].reshape(-1), v[1:].reshape(-1)])
    g = gbx.graph_build(n, s, d)
    x, y = torch.arange(w, device="cuda"), torch.arange(h, device="cuda")
    for sx, sy in ((w // 2, h // 2), (0, h - 1)):
        src = sy * w + sx
        want = ((y - sy).abs()[:, None] + (x - sx).abs()[None, :]).to(torch.int32).view(-1)
        depth, parent = run(g, n, src, gbx.desc_init())
        assert torch.equal(depth, want)
        assert int(parent[src]) == src
        p = parent.long()
        ids = torch.arange(n, device="cuda")
        rest = ids != src
        assert bool((torch.abs(p // w - ids // w) + torch.abs(p % w - ids % w) == 1)[rest].all())
        assert bool((want[p] == want - 1)[rest].all())
    g.free()


@pytest.mark.parametrize("fanout", [2, 20, 31])
@pytest.mark.parametrize("directed", [False, True])
def test_tree_handed_over(fanout, directed):
    n = 8_000_003
    d = torch.arange(1, n, dtype=torch.int64, device="cuda")
    up = (d - 1) // fanout
    g = gbx.graph_build(n, up.to(torch.int32), d.to(torch.int32), symmetrize=not directed)
    want, size, first, level = torch.empty(n, dtype=torch.int32, device="cuda"), 1, 0, 0
    while first < n:
        want[first:first + size] = level
        first, size, level = first + size, size * fanout, level + 1
    for desc in (gbx.desc_init(), gbx.desc_init(direction=gbx.DIR_PUSH)):
        depth, parent = run(g, n, 0, desc)
        assert torch.equal(depth, want)
        assert int(parent[0]) == 0 and torch.equal(parent[1:].long(), up)
    g.free()
