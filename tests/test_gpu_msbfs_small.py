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
