"""The power iteration as one launch (small and medium problems): the norms against the
oracle's power iteration of the same scaled problem, at the 1e-9 of the other norm tests,
and the same bits from one preparation to the next."""
import numpy as np
import pytest

from oracle import pdhg as O
from synth import instance_seed, lp_instance, qp_instance, qp_sparse_q_instance
from tests.gpu_util import lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    return lib()


CASES = {
    # one CTA; a few; all SMs with the partials added by every CTA; chunk sums (more than
    # 2048 items); sliced rows; F^T with 32 long rows; a general Q (one product a round)
    "one_cta": lambda: lp_instance(60, 120, seed=instance_seed(301), density=0.05),
    "few_ctas": lambda: lp_instance(800, 1500, seed=instance_seed(302), density=0.01),
    "all_sms": lambda: lp_instance(6000, 9000, seed=instance_seed(303), density=0.003),
    "chunk_sums": lambda: lp_instance(30000, 50000, seed=instance_seed(304), nnz=700000,
                                      rows="zipf"),
    "qp": lambda: qp_instance(20000, 10000, seed=instance_seed(305), a_density=1e-3, f_cols=32,
                              f_density=0.01),
    "sparse_q": lambda: qp_sparse_q_instance(3000, 1200, seed=instance_seed(306),
                                             a_density=2e-3, b_density=1e-3),
}


@pytest.mark.parametrize("case", list(CASES))
def test_single_launch_norms_match_oracle(C, case):
    from paper_2412_09734_gb300.problem import Problem
    d = CASES[case]()
    p = Problem.from_dict(d)
    norms = []
    for _ in range(2):
        C.mpax_prepare(p.h, C.mpax_options_default())
        info = C.mpax_get_scaling(p.h, d["m"], d["n"])[2]
        norms.append((info["norm_A"], info["norm_Q"]))
    p.close()
    assert norms[0] == norms[1]
    _, _, _, nA, nQ, _, _ = O.prepare(O.problem_from_arrays(d), O.Options())
    np.testing.assert_allclose(norms[0][0], nA, rtol=1e-9)
    if p.is_qp:
        np.testing.assert_allclose(norms[0][1], nQ, rtol=1e-9)


@pytest.mark.parametrize("rows", [16_800_000, 16_700_000])
def test_norm_sum_over_very_many_items(C, rows):
    """0.7 times the identity: every work item (64 rows) adds alike to the norm of the first
    round, on both sides of the 262,144 items from which all warps of a block share the sum."""
    import torch
    n = rows
    rp = torch.arange(n + 1, dtype=torch.int64, device="cuda")
    col = torch.arange(n, dtype=torch.int32, device="cuda")
    one = torch.ones(n, dtype=torch.float64, device="cuda")
    h = C.mpax_lp_create(n, n, rp, col, 0.7 * one, one, one, one, 0 * one, one)
    try:
        C.mpax_prepare(h, C.mpax_options_default(ruiz_iters=0, pock_chambolle=0, spmv_kernel=0))
        _, _, info = C.mpax_get_scaling(h, n, n)
    finally:
        C.mpax_destroy(h)
    np.testing.assert_allclose(info["norm_A"], 0.7, rtol=1e-12)


@pytest.mark.parametrize("case", list(CASES))
def test_short_rounds_run_and_agree_with_the_general_kernels(C, case):
    """A caller that names the kernel of the products gets the rounds of the general kernels:
    the same norms to the 1e-9 of the oracle's, and more launches in all (four a round against
    at most two and one at the end, in four rounds or more)."""
    from paper_2412_09734_gb300.problem import Problem
    d = CASES[case]()
    p = Problem.from_dict(d)
    got = {}
    for kind in (-1, -1, 0):  # the first solve also times the kernels
        C.mpax_solve(p.h, C.mpax_options_default(spmv_kernel=kind, iteration_limit=64, eps_abs=1e-14,
                                                 eps_rel=1e-14))
        info = C.mpax_get_scaling(p.h, d["m"], d["n"])[2]
        got[kind] = (info["norm_A"], info["norm_Q"], C.mpax_get_stats(p.h)["kernel_launches"])
    p.close()
    np.testing.assert_allclose(got[-1][0], got[0][0], rtol=1e-9)
    if p.is_qp:
        np.testing.assert_allclose(got[-1][1], got[0][1], rtol=1e-9)
    assert got[0][2] >= got[-1][2] + 7 * (2 if p.is_qp else 1)
