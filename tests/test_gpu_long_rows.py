"""Rows of more than 64 entries in the scaling: they come from a list of their own, a warp
each, whether they stand together (the coupling rows of a model) or apart."""
import time

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


def _create(C, A):
    m, n = A.shape
    return C.mpax_lp_create(m, n, A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data,
                            np.ones(n), np.zeros(m), np.ones(m), np.zeros(n), np.ones(n))


def _matrix(lengths, n, seed):
    rng = np.random.default_rng(seed)
    cols = [np.sort(rng.choice(n, size=k, replace=False)) for k in lengths]
    val = rng.standard_normal(sum(lengths)) * 10.0 ** rng.uniform(-3, 3, sum(lengths))
    return sp.csr_matrix((val, np.concatenate(cols), np.concatenate([[0], np.cumsum(lengths)])),
                         shape=(len(lengths), n))


# all rows long, fewer and more of them than a block's warps; long rows at both ends of a
# warp's four and of the matrix; and the same for columns (the transpose)
@pytest.mark.parametrize("lengths,n", [
    ([200] * 3, 500),
    ([90] * 21, 300),
    ([65] * 10000, 400),
    ([300, 300] + [2] * 700 + [64, 65] * 9 + [400] * 13, 600),
])
@pytest.mark.parametrize("transposed", [False, True])
def test_scaling_of_long_rows_matches_oracle(C, lengths, n, transposed):
    A = _matrix(lengths, n, n)
    A = sp.csr_matrix(A.T) if transposed else A
    A.sort_indices()
    h = _create(C, A)
    try:
        for _ in range(2):
            C.mpax_prepare(h, C.mpax_options_default(power_max_iter=0))
            Dr, Dc, _ = C.mpax_get_scaling(h, *A.shape)
            rDr, rDc = O.scaling_factors(A, 10, True, None)
            np.testing.assert_allclose(Dr, rDr, rtol=1e-12)
            np.testing.assert_allclose(Dc, rDc, rtol=1e-12)
    finally:
        C.mpax_destroy(h)


def test_long_rows_side_by_side_cost_what_they_cost_apart(C):
    """20 rows of 100,000 entries next to one another and with three empty rows between."""
    import torch
    m, n, k = 20, 300000, 100000
    rng = np.random.default_rng(1)
    col = np.concatenate([3 * np.arange(k) + r % 3 for r in range(m)])
    val = rng.standard_normal(m * k)
    best = {}
    for gap in (1, 4):
        rp = np.zeros(gap * m + 1, dtype=np.int64)
        rp[1:] = k * ((np.arange(gap * m) + gap) // gap)
        h = _create(C, sp.csr_matrix((val, col, rp), shape=(gap * m, n)))
        try:
            ts = []
            for _ in range(5):
                torch.cuda.synchronize()
                t = time.perf_counter()
                C.mpax_prepare(h, C.mpax_options_default(power_max_iter=0))
                torch.cuda.synchronize()
                ts.append(time.perf_counter() - t)
        finally:
            C.mpax_destroy(h)
        best[gap] = min(ts)
    assert best[1] <= 1.5 * best[4]
