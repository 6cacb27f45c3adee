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
