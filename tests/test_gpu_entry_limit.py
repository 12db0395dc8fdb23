"""Rows whose entries are the last of 2^31 - 1: the pull's positions past a row's end do not fit
32 bits.  The column array is given by an address that many entries before its first one in
memory; only its end exists and is read."""
import numpy as np
import pytest

from paper_1804_03327_gb300 import gbx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LAST = 2**31 - 1  # one past the last entry a graph can hold


@pytest.mark.parametrize("early_exit", [0, 1])
@pytest.mark.parametrize("density", [0.0, 0.001, 0.4])
@pytest.mark.parametrize("last", [1, 3, 7, 17, 20, 150, 1040, 1041, 1100, 5000, 9000])
def test_rows_at_the_entry_limit(last, density, early_exit):
    rng = np.random.default_rng(last)
    n = 5000
    lengths = np.zeros(n, np.int64)
    lengths[[0, 40, 41, 63, 700]] = 5, 1500, 33, 2, 18
    lengths[n - 1] = last
    ptr = LAST - lengths.sum() + np.concatenate([[0], np.cumsum(lengths)])
    col = rng.integers(0, n, lengths.sum()).astype(np.int32)
    u = (rng.random(n) < density).astype(np.uint8)
    ptr_d = torch.from_numpy(ptr.astype(np.int32)).cuda()
    pad = torch.zeros(8, dtype=torch.int32, device="cuda")
    col_d = torch.cat([torch.from_numpy(col).cuda(), pad])
    u_d, w = torch.from_numpy(u).cuda(), torch.full((n,), 7, dtype=torch.uint8, device="cuda")
    base = col_d.data_ptr() - 4 * int(ptr[0])
    assert base > 0 and ptr[-1] == LAST
    gbx.mxv_pull_noalloc(n, ptr_d.data_ptr(), base, u_d, None, w, False, bool(early_exit))
    torch.cuda.synchronize()
    want = np.array([u[col[a:b]].any() for a, b in zip(ptr[:-1] - ptr[0], ptr[1:] - ptr[0])], np.uint8)
    assert np.array_equal(w.cpu().numpy(), want)
