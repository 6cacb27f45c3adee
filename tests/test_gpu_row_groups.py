"""Row-wise preprocessing kernels at the edges of their lane groups: the scaling takes
rows of up to 64 entries eight lanes each, four rows to a warp, and longer ones with
the whole warp; the transpose sorts long rows of A^T a few to a CTA, in shared memory up
to 4096 entries.  Scaling factors against the oracle's, transposes against scipy's."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import pdhg as O
from tests.gpu_util import lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    return lib()


def _matrix(lengths, n, seed):
    rng = np.random.default_rng(seed)
    cols = [np.sort(rng.choice(n, size=k, replace=False)) for k in lengths]
    rp = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    col = np.concatenate(cols).astype(np.int32) if rp[-1] else np.empty(0, np.int32)
    val = rng.standard_normal(int(rp[-1])) * 10.0 ** rng.uniform(-3, 3, int(rp[-1]))
    return rp, col, val


@pytest.mark.parametrize("lengths,n", [
    ([1], 1),
    ([0, 7, 8, 9, 31], 40),                      # a warp's rows and one more
    ([32, 33, 63, 64, 65, 66, 0, 200, 64], 300),  # both sides of the group limit in one warp
    ([300, 1, 300, 1, 1, 1, 300], 400),
    ([2] * 5001, 3),                              # three rows of A^T of about 3,300 entries
    ([1] * 9000, 2),                              # two of about 4,500: sorted in global memory
])
def test_scaling_and_transpose_at_row_group_edges(C, lengths, n):
    m = len(lengths)
    rp, col, val = _matrix(lengths, n, m + n)
    A = sp.csr_matrix((val, col, rp), shape=(m, n))
    h = C.mpax_lp_create(m, n, rp, col, val, np.ones(n), np.zeros(m), np.ones(m), np.zeros(n),
                         np.ones(n))
    try:
        C.mpax_prepare(h, C.mpax_options_default(power_max_iter=0))
        Dr, Dc, _ = C.mpax_get_scaling(h, m, n)
        trp, tcol, tval = C.mpax_get_transpose(h, n, len(val))
    finally:
        C.mpax_destroy(h)
    rDr, rDc = O.scaling_factors(A, 10, True, None)
    np.testing.assert_allclose(Dr, rDr, rtol=1e-12)
    np.testing.assert_allclose(Dc, rDc, rtol=1e-12)
    At = A.T.tocsr()
    At.sort_indices()
    np.testing.assert_array_equal(trp, At.indptr)
    np.testing.assert_array_equal(tcol, At.indices)
    np.testing.assert_array_equal(tval, At.data)


# The work items of a product hold at most 64 short rows and start a new one at a multiple
# of 64 only where rows are short: runs of empty rows, rows of 3 to 5 entries (on both
# sides of 256 entries per 64 and per 32 rows), of 8 and of 40, and bursts of either.  Every
# row's product at 1e-12 through one iteration in FP64 (a lost or doubled row is wrong
# altogether; the sums themselves are good to 1e-14).
@pytest.mark.parametrize("pattern", ["empty", "three", "four", "mixed8", "forty", "bursts"])
def test_packed_items_cover_every_row_once(C, pattern):
    rng = np.random.default_rng(len(pattern))
    m, n = 1300, 900
    lengths = {"empty": np.where(np.arange(m) % 400 < 330, 0, 5),
               "three": np.full(m, 3), "four": rng.integers(3, 6, m),
               "mixed8": rng.integers(4, 13, m), "forty": np.full(m, 40),
               "bursts": np.where((np.arange(m) // 70) % 2 == 0, 0, 60)}[pattern]
    rp, col, val = _matrix(list(lengths), n, 77)
    A = sp.csr_matrix((val, col, rp), shape=(m, n))
    h = C.mpax_lp_create(m, n, rp, col, val, np.ones(n), np.full(m, -np.inf), np.zeros(m),
                         np.full(n, -1e30), np.full(n, 1e30))
    try:
        C.mpax_prepare(h, C.mpax_options_default(ruiz_iters=0, pock_chambolle=0, power_max_iter=2))
        x, y = rng.standard_normal(n), rng.standard_normal(m)
        C.mpax_set_iterate(h, x, y, x, y, 0, 1.0, 1.0)
        C.mpax_iterate(h, 1)
        _, _, xh, yh = C.mpax_get_iterate(h, m, n)
    finally:
        C.mpax_destroy(h)
    np.testing.assert_allclose(xh, x - (1.0 - A.T @ y), rtol=1e-12, atol=1e-12 * np.abs(val).sum())
    v = y - A @ (2 * xh - x)  # y^ = v - proj_[0, inf)(v)
    np.testing.assert_allclose(yh, np.minimum(v, 0.0), rtol=1e-12,
                               atol=1e-12 * np.abs(val).sum())


# The same patterns with equality rows: y^ = v - proj(v) = v shows the product of every row,
# and of every column through x^, against a bound of its own.  A row sum of at most 100 terms
# in FP64 is good to 1.2e-14 of the sum of their magnitudes, and x^ enters the rows' products
# with that error once more; 1e-13 of the magnitudes is far below a lost or doubled entry.
@pytest.mark.parametrize("pattern", ["empty", "three", "four", "mixed8", "forty", "bursts"])
def test_every_row_and_column_product(C, pattern):
    rng = np.random.default_rng(len(pattern))
    m, n = 1300, 900
    lengths = {"empty": np.where(np.arange(m) % 400 < 330, 0, 5),
               "three": np.full(m, 3), "four": rng.integers(3, 6, m),
               "mixed8": rng.integers(4, 13, m), "forty": np.full(m, 40),
               "bursts": np.where((np.arange(m) // 70) % 2 == 0, 0, 60)}[pattern]
    rp, col, val = _matrix(list(lengths), n, 78)
    A = sp.csr_matrix((val, col, rp), shape=(m, n))
    assert max(np.diff(rp).max(), np.bincount(col).max()) <= 100
    h = C.mpax_lp_create(m, n, rp, col, val, np.ones(n), np.zeros(m), np.zeros(m),
                         np.full(n, -1e30), np.full(n, 1e30))
    try:
        C.mpax_prepare(h, C.mpax_options_default(ruiz_iters=0, pock_chambolle=0, power_max_iter=2))
        x, y = rng.standard_normal(n), rng.standard_normal(m)
        C.mpax_set_iterate(h, x, y, x, y, 0, 1.0, 1.0)
        C.mpax_iterate(h, 1)
        _, _, xh, yh = C.mpax_get_iterate(h, m, n)
    finally:
        C.mpax_destroy(h)
    ref = x - (1.0 - A.T @ y)
    bx = 1e-13 * (np.abs(x) + 1.0 + abs(A).T @ np.abs(y))
    assert np.all(np.abs(xh - ref) <= bx)
    by = 1e-13 * np.abs(y) + abs(A) @ (1e-13 * np.abs(x) + 3.0 * bx)
    assert np.all(np.abs(yh - (y - A @ (2.0 * ref - x))) <= by)
