"""The (min, +) pull where its form changes with the rows' lengths: a lane per row, groups of 1, 4 and
8 lanes, and one row around the length from which it is deferred -- called directly, after AUTO has
counted u, and again on the scratch that the call before left.  Equal to the oracle's float64 result
rounded once."""
import numpy as np
import pytest

import oracle
from paper_1804_03327_gb300 import gbx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N = 3001


def graph(k, longest, N=N):
    """Every vertex has edges to the k next ones; vertex 5 has `longest` in-edges from elsewhere."""
    s = np.repeat(np.arange(N, dtype=np.int32), k)
    d = ((s + np.tile(np.arange(1, k + 1, dtype=np.int32), N)) % N).astype(np.int32)
    keep = d != 5
    hub = np.random.default_rng(longest).permutation(np.arange(100, N, dtype=np.int32))[:longest]
    s, d = np.concatenate([s[keep], hub]), np.concatenate([d[keep], np.full(longest, 5, np.int32)])
    return s.astype(np.int32), d.astype(np.int32)


@pytest.mark.parametrize("k,longest", [(4, 3), (4, 20), (4, 21), (4, 32), (4, 33), (4, 512 + 4), (4, 2000),
                                       (8, 80), (8, 81), (8, 700), (16, 160), (16, 161), (16, 2500), (30, 0)])
@pytest.mark.parametrize("transpose", [0, 1])
def test_row_lengths(k, longest, transpose, N=N):
    s, d = graph(k, longest, N)
    rng = np.random.default_rng(k)
    val = rng.random(len(s)).astype(np.float32)
    og = oracle.graph_weighted(N, s, d, val, symmetrize=False)
    g = gbx.graph_build(N, s, d, symmetrize=False)
    gbx.graph_set_weights(g, s, d, val)
    u = np.where(rng.random(N) < 0.4, (rng.random(N) * 9).astype(np.float32), np.float32(np.inf))
    m = (rng.random(N) < 0.6).astype(np.uint8)
    old = np.where(rng.random(N) < 0.5, (rng.random(N) * 3).astype(np.float32), np.float32(np.inf))
    u_d, m_d = torch.from_numpy(u).cuda(), torch.from_numpy(m).cuda()
    for masked, complement, accum in ((0, 0, 0), (1, 0, 0), (1, 1, 1), (0, 0, 1), (1, 1, 0), (0, 1, 1), (0, 1, 0)):
        want = oracle.mxv_minplus(N, N, og.out_ptr, og.out_col, og.out_val, u.astype(np.float64),
                                  m if masked else None, transpose=bool(transpose), complement=bool(complement),
                                  accum=bool(accum), w_old=old.astype(np.float64)).astype(np.float32)
        for direction in (gbx.DIR_PULL, gbx.DIR_AUTO, gbx.DIR_PULL, gbx.DIR_PUSH, gbx.DIR_PULL):
            w = torch.from_numpy(old.copy()).cuda()
            gbx.mxv(gbx.dense_f32(w), gbx.dense(m_d) if masked else None, gbx.MIN_PLUS_F32, g, gbx.dense_f32(u_d),
                    gbx.desc_init(direction=direction, transpose=transpose, mask_complement=complement, accum=accum,
                                  alpha=0.01))
            assert np.array_equal(w.cpu().numpy(), want), (masked, complement, accum, direction)
    g.free()


@pytest.mark.parametrize("n", [5003, 14401, 60001])
@pytest.mark.parametrize("k,longest", [(4, 20), (4, 21), (4, 33), (4, 600), (7, 80), (7, 81), (16, 160), (16, 161),
                                       (16, 320), (16, 321), (5, 640), (5, 2176), (5, 2177), (5, 4000)])
def test_row_lengths_by_group_width(n, k, longest):
    """More vertices: fewer lanes a row."""
    test_row_lengths(k, longest, 1, n)


@pytest.mark.parametrize("longest", [2000, 16384, 16385, 24000])
@pytest.mark.parametrize("visited", [0.0, 0.9])
def test_many_long_rows(longest, visited):
    """More long rows in one block than it keeps (neighbouring rows), and rows around the length from
    which they are left to the grid."""
    n, hubs = 40000, 700
    r = np.random.default_rng(longest)
    lengths = np.full(hubs, 300)
    lengths[::50] = longest
    d = np.repeat(np.arange(hubs), lengths)
    s = np.concatenate([r.permutation(np.arange(hubs, n))[:x] for x in lengths])
    s, d = s.astype(np.int32), d.astype(np.int32)
    val = r.random(len(s)).astype(np.float32)
    og = oracle.graph_weighted(n, s, d, val, symmetrize=False)
    g = gbx.graph_build(n, s, d, symmetrize=False)
    gbx.graph_set_weights(g, s, d, val)
    u = np.where(r.random(n) < 0.02, (r.random(n) * 9).astype(np.float32), np.float32(np.inf))
    m = (r.random(n) < visited).astype(np.uint8)
    old = (r.random(n) * 3).astype(np.float32)
    u_d, m_d = torch.from_numpy(u).cuda(), torch.from_numpy(m).cuda()
    for accum in (0, 1):
        want = oracle.mxv_minplus(n, n, og.out_ptr, og.out_col, og.out_val, u.astype(np.float64), m, transpose=True,
                                  complement=True, accum=bool(accum), w_old=old.astype(np.float64)).astype(np.float32)
        for _ in range(2):
            w = torch.from_numpy(old.copy()).cuda()
            gbx.mxv(gbx.dense_f32(w), gbx.dense(m_d), gbx.MIN_PLUS_F32, g, gbx.dense_f32(u_d),
                    gbx.desc_init(direction=gbx.DIR_PULL, mask_complement=1, accum=accum))
            assert np.array_equal(w.cpu().numpy(), want), accum
    g.free()
