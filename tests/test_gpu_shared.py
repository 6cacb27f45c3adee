"""GPU parity of the shared-matrix dense batch (tensor-core BF16x3 products and
the FP32 product path) against the FP64 oracle on each instance."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import pdhg as O
from synth import shared_dense_lp_batch
from tests.gpu_util import lib, rel_inf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    return lib()


def _oracle_problem(d, k):
    A = sp.csr_matrix(d["A"].astype(np.float64))
    return O.Problem(A, d["C"][k].copy(), d["b"].copy(), d["b"].copy(), d["l"], d["u"])


# On the fully degenerate construction (s = 0, bound_frac = 0) the BF16x3 rounding
# lets x drift along the optimal face and the primal-weight rule drives omega to
# ~1e-4 for about half of the instances (reproduced on the CPU by rounding the
# oracle's products the same way); those instances stall, and the solve continues
# with FP32 products.
@pytest.mark.parametrize("fp32,bound_frac", [(False, 0.5), (False, 0.0), (True, 0.0)])
def test_shared_batch_matches_oracle(C, fp32, bound_frac):
    d = shared_dense_lp_batch(192, 384, 24, seed=31337, bound_frac=bound_frac)
    h = C.mpax_lp_shared_create(d["m"], d["n"], d["B"], d["A"], d["C"], d["b"], d["b"],
                                d["l"], d["u"])
    try:
        C.mpax_shared_solve(h, C.mpax_options_default(eps_abs=1e-4, eps_rel=1e-4,
                                                      iteration_limit=200000), fp32)
        summ, per = C.mpax_shared_get_stats(h, d["B"])
        X, Y = C.mpax_shared_get_solution(h, d["m"], d["n"], d["B"])
    finally:
        C.mpax_shared_destroy(h)
    assert summ["n_optimal"] == d["B"]
    assert summ["gemms"] > 0 and summ["gemm_flops"] > 0
    if fp32:
        assert summ["fp64_instances"] == 0
    for k in range(d["B"]):
        p = _oracle_problem(d, k)
        chk = O.kkt(p, X[k], Y[k])
        assert chk["converged"], (k, chk["rel_kkt"])
        # literal construction: every feasible point is optimal with value c^T x0
        assert chk["primal_obj"] == pytest.approx(d["opt_value"][k], rel=1e-3, abs=1e-3)
    # the same instance through the single-problem FP64 path of the oracle
    ref = O.solve_lp(_oracle_problem(d, 0), O.Options())
    assert ref.kkt["primal_obj"] == pytest.approx(d["opt_value"][0], rel=1e-3, abs=1e-3)


def test_shared_nondegenerate_values(C):
    """Costs with reduced-cost parts at bounds (unique optimum): values to 1e-4."""
    d = shared_dense_lp_batch(128, 256, 8, seed=99)
    rng = np.random.default_rng(7)
    X0 = rng.uniform(0, 1, size=(d["B"], d["n"]))
    S = np.zeros_like(X0)
    at_l = rng.random(X0.shape) < 0.3
    at_u = (~at_l) & (rng.random(X0.shape) < 0.43)
    X0[at_l], X0[at_u] = 0.0, 1.0
    S[at_l] = rng.uniform(0.1, 1.0, at_l.sum())
    S[at_u] = -rng.uniform(0.1, 1.0, at_u.sum())
    # a common equality right-hand side needs a common x0; keep the one of the batch
    # and only add reduced-cost parts at the bounds of that shared x0
    x0 = d["x0"].copy()
    lo = rng.random(d["n"]) < 0.3
    hi = (~lo) & (rng.random(d["n"]) < 0.43)
    x0[lo], x0[hi] = 0.0, 1.0
    b = d["A"].astype(np.float64) @ x0
    Cm = d["Y"] @ d["A"].astype(np.float64)
    Cm[:, lo] += rng.uniform(0.1, 1.0, (d["B"], lo.sum()))
    Cm[:, hi] -= rng.uniform(0.1, 1.0, (d["B"], hi.sum()))
    h = C.mpax_lp_shared_create(d["m"], d["n"], d["B"], d["A"], Cm, b, b, d["l"], d["u"])
    try:
        C.mpax_shared_solve(h, C.mpax_options_default(iteration_limit=200000))
        summ, per = C.mpax_shared_get_stats(h, d["B"])
        X, Y = C.mpax_shared_get_solution(h, d["m"], d["n"], d["B"])
    finally:
        C.mpax_shared_destroy(h)
    assert summ["n_optimal"] == d["B"]
    for k in range(d["B"]):
        p = O.Problem(sp.csr_matrix(d["A"].astype(np.float64)), Cm[k], b, b, d["l"], d["u"])
        chk = O.kkt(p, X[k], Y[k])
        assert chk["converged"]
        assert chk["primal_obj"] == pytest.approx(float(Cm[k] @ x0), rel=1e-3, abs=1e-3)


def test_shared_values_autograd(C):
    """d v_k / d c_k = x_k*: the backward of the value layer returns the solved
    primal rows, whose values match c_k^T x0 and whose KKT error the oracle checks."""
    import torch
    from paper_2412_09734_gb300.autograd import SharedFeasibleSet, SharedLPValues
    # 3/4 of x0 on a bound leaves ~32 free coordinates against 64 equality rows:
    # a tall, well-conditioned system, so x0 is the unique optimum
    d = shared_dense_lp_batch(64, 128, 6, seed=4242, bound_frac=0.75)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    Cm = dev(d["C"]).requires_grad_(True)
    w = torch.linspace(0.5, 1.5, d["B"], dtype=torch.float64, device="cuda")
    fs = SharedFeasibleSet(dev(d["A"]), dev(d["b"]), dev(d["b"]), dev(d["l"]), dev(d["u"]),
                           d["B"])
    v = SharedLPValues.apply(Cm, fs, dict(eps_abs=1e-4, eps_rel=1e-4, iteration_limit=400000))
    (w * v).sum().backward()
    np.testing.assert_allclose(v.detach().cpu().numpy(), d["opt_value"], rtol=1e-3, atol=1e-3)
    G = Cm.grad.cpu().numpy()
    for k in range(d["B"]):
        xk = G[k] / float(w[k])
        p = O.Problem(sp.csr_matrix(d["A"].astype(np.float64)), d["C"][k].copy(), d["b"],
                      d["b"], d["l"], d["u"])
        chk = O.kkt(p, xk, np.zeros(d["m"]))
        assert chk["primal_res"] / (1 + chk["b_norm"]) <= 1e-4
        # x0 is the unique optimum, so the gradient row is x0 up to the solve tolerance
        np.testing.assert_allclose(xk, d["x0"], atol=5e-3)


def test_spo_plus_loss_matches_oracle(C):
    """SPO+ over a shared feasible set: the batched losses equal the oracle's, and
    the returned gradient rows are subgradients of the oracle's loss (convexity
    inequality along random directions)."""
    import torch
    from oracle import spo
    from paper_2412_09734_gb300.autograd import SharedFeasibleSet, SharedLPValues, SPOPlusLoss
    d = shared_dense_lp_batch(64, 128, 4, seed=777, bound_frac=0.75)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    opts = dict(eps_abs=1e-6, eps_rel=1e-6, iteration_limit=400000)
    A, b, l, u = dev(d["A"]), dev(d["b"]), dev(d["l"]), dev(d["u"])
    fs = SharedFeasibleSet(A, b, b, l, u, d["B"])
    Ct = dev(d["C"])
    with torch.no_grad():
        zt = SharedLPValues.apply(Ct, fs, opts, True)
    # the true optimum is x0 (unique, reduced costs at the bounds)
    Xt = torch.from_numpy(np.tile(d["x0"], (d["B"], 1))).cuda()
    rng = np.random.default_rng(11)
    Ch = dev(d["C"] + rng.normal(0, 0.5, d["C"].shape)).requires_grad_(True)
    loss = SPOPlusLoss.apply(Ch, Ct, Xt, zt, fs, opts, True)
    loss.sum().backward()
    G = Ch.grad.cpu().numpy()
    Lg = loss.detach().cpu().numpy()
    Ah = sp.csr_matrix(d["A"].astype(np.float64))
    oo = O.Options(eps_abs=1e-8, eps_rel=1e-8, iteration_limit=10**6)
    for k in range(d["B"]):
        p = O.Problem(Ah, d["C"][k].copy(), d["b"], d["b"], d["l"], d["u"])
        ch = Ch.detach().cpu().numpy()[k]
        # the oracle side takes the closed-form optimum c_k^T x0 of the construction
        lo, go, _ = spo.spo_plus(p, ch, d["x0"], float(d["opt_value"][k]), oo)
        assert Lg[k] == pytest.approx(lo, rel=1e-3, abs=1e-3)
        for _ in range(3):
            delta = rng.normal(0, 0.1, d["n"])
            l2 = spo.spo_plus(p, ch + delta, d["x0"], float(d["opt_value"][k]), oo)[0]
            assert l2 >= lo + G[k] @ delta - 1e-3 * (1 + abs(lo))


def test_dense_single_knapsack_matches_highs(C):
    """One dense LP (the knapsack relaxation, B = 1, FP32 products: with one cost
    vector the products are matrix-vector products) against HiGHS's optimum and
    the oracle's KKT evaluation."""
    from scipy.optimize import linprog
    from synth import knapsack_lp
    d = knapsack_lp(40, 2000, seed=2024)
    h = C.mpax_lp_shared_create(d["d"], d["m_items"], 1, d["A"], d["c"][None, :], d["lc"],
                                d["uc"], d["l"], d["u"])
    try:
        C.mpax_shared_solve(h, C.mpax_options_default(eps_abs=1e-6, eps_rel=1e-6,
                                                      iteration_limit=400000), True)
        summ, per = C.mpax_shared_get_stats(h, 1)
        X, Y = C.mpax_shared_get_solution(h, d["d"], d["m_items"], 1)
    finally:
        C.mpax_shared_destroy(h)
    assert summ["n_optimal"] == 1
    A = d["A"].astype(np.float64)
    p = O.Problem(sp.csr_matrix(A), d["c"], d["lc"], d["uc"], d["l"], d["u"])
    chk = O.kkt(p, X[0], Y[0], 1e-6, 1e-6)
    assert chk["converged"], chk["rel_kkt"]
    res = linprog(d["c"], A_ub=A, b_ub=d["uc"], bounds=(0, 1), method="highs")
    assert res.status == 0
    assert chk["primal_obj"] == pytest.approx(res.fun, rel=1e-5)


@pytest.fixture(scope="module")
def iterate_case():
    """A shared batch whose products span several tiles with ragged edges in every
    dimension (m = 2036 rows and n = 4100 columns are not multiples of the 128-row
    output tile or the 32-wide K block; 500 instances fill one 256-wide instance
    tile and part of a second), and the oracle's point after 192 iterations for
    the first and last instance of each instance tile."""
    d = shared_dense_lp_batch(2036, 4100, 500, seed=2412, bound_frac=0.5)
    A = sp.csr_matrix(d["A"].astype(np.float64))
    k_iter = 192
    ref = {}
    for k in (0, 255, 256, 499):
        p = O.Problem(A, d["C"][k].copy(), d["b"].copy(), d["b"].copy(), d["l"], d["u"])
        ref[k] = O.solve_lp(p, O.Options(eps_abs=1e-14, eps_rel=1e-14, iteration_limit=k_iter,
                                         power_max_iter=0, eps_primal_infeasible=0.0,
                                         eps_dual_infeasible=0.0))
        assert ref[k].iterations == k_iter and ref[k].status == "iteration_limit"
    assert any(r.restarts > 0 for r in ref.values())
    return d, k_iter, ref


# Tolerances.  The FP32 product path rounds the scaled matrix, the iterates and
# every product to FP32; the mixed-precision batch kernel meets 1e-5 after 64
# iterations, and 192 iterations with two restarts take 2e-5.  The BF16x3 path
# forms each product from the split operands, which keep 2^-17 relative error
# per element, and accumulates in FP32 on the tensor cores, whose error grows
# with the length K of the sums (the (3K + 2) 2^-24 term of the product's stated
# bound; on the 16384 x 32768 matrix of the dense bench the normwise product
# error is 1.1e-4 at K = 32768, about 1.4e-5 when scaled to K = 4100).  Modelling
# the split's rounding in FP64 on the CPU moves the oracle's point at iteration
# 192 by 1.5e-5 here; 2e-4 leaves room for the accumulation, while a product
# that drops one of its three terms (A_lo v_hi, say) moves the same point by
# 3e-3 after only 64 iterations in that model.
@pytest.mark.parametrize("fp32,tol", [(False, 2e-4), (True, 2e-5)], ids=["bf16x3", "fp32"])
def test_shared_iterates_match_oracle(C, iterate_case, fp32, tol):
    """Iterate-level parity of the shared-matrix batch (eqs. 3-4, Algorithm 1 per
    column): 192 iterations from zero, with their checks, restarts and
    primal-weight updates, give the oracle's (x^, y^) element by element for the
    instances at the edges of both instance tiles, with the step sizes from the
    certified bound ||A~||_2 <= 1 on both sides."""
    d, k_iter, ref = iterate_case
    h = C.mpax_lp_shared_create(d["m"], d["n"], d["B"], d["A"], d["C"], d["b"], d["b"],
                                d["l"], d["u"])
    try:
        C.mpax_shared_solve(h, C.mpax_options_default(eps_abs=1e-14, eps_rel=1e-14,
                                                      iteration_limit=k_iter, power_max_iter=0,
                                                      fp64_continuation=0), fp32)
        summ, per = C.mpax_shared_get_stats(h, d["B"])
        X, Y = C.mpax_shared_get_solution(h, d["m"], d["n"], d["B"])
    finally:
        C.mpax_shared_destroy(h)
    assert np.all(per["iterations"] == k_iter)
    assert summ["fp64_instances"] == 0
    assert summ["gemms"] > 0
    for k, r in ref.items():
        assert rel_inf(X[k], r.x) <= tol, (k, rel_inf(X[k], r.x))
        assert rel_inf(Y[k], r.y) <= tol, (k, rel_inf(Y[k], r.y))


# The scaling rounds run over tiles of 64 rows by 256 columns (n % 4 != 0) or 1024: one
# element, one short of a tile, one over, and several tiles of each kind.  `spread`
# scales rows and columns by up to 10^+-spread, past the range in which the scaled
# value is formed from float pairs (spread 12: factors near 1e-12 on values near 1e24).
# 64 iterations in FP32 products as in test_shared_iterates_match_oracle: 1e-5.
@pytest.mark.parametrize("m,n,spread", [(1, 1, 0), (63, 255, 0), (65, 257, 0), (64, 1024, 0),
                                        (130, 1028, 3), (70, 515, 12)])
def test_shared_scaling_tiles_match_oracle(C, m, n, spread):
    rng = np.random.default_rng(m * 1000 + n)
    A = rng.standard_normal((m, n)) / np.sqrt(n)
    A[rng.random((m, n)) < 0.1] = 0.0
    A *= 10.0 ** rng.uniform(-spread, spread, (m, 1)) * 10.0 ** rng.uniform(-spread, spread, n)
    A = A.astype(np.float32)
    A64 = A.astype(np.float64)
    x0 = rng.uniform(0, 1, n)
    b, c = A64 @ x0, A64.T @ (rng.standard_normal((2, m)) / np.maximum(np.abs(A64).max(1), 1e-300)).T
    p = O.Problem(sp.csr_matrix(A64), c[:, 1].copy(), b, b, np.zeros(n), np.ones(n))
    opts = dict(eps_abs=1e-14, eps_rel=1e-14, iteration_limit=64, power_max_iter=0)
    ref = O.solve_lp(p, O.Options(eps_primal_infeasible=0.0, eps_dual_infeasible=0.0, **opts))
    h = C.mpax_lp_shared_create(m, n, 2, A, np.ascontiguousarray(c.T), b, b, np.zeros(n), np.ones(n))
    try:
        C.mpax_shared_solve(h, C.mpax_options_default(fp64_continuation=0, **opts), True)
        X, Y = C.mpax_shared_get_solution(h, m, n, 2)
    finally:
        C.mpax_shared_destroy(h)
    # in the scaled space, where every coordinate has the same weight
    assert rel_inf(X[1] / ref.Dc, ref.x / ref.Dc) <= 1e-5
    assert rel_inf(Y[1] / ref.Dr, ref.y / ref.Dr) <= 1e-5


# The FP32 products pick a tile by the size of the grid: 32 x 32 outputs, 64 x 32 from 128
# tiles on, 128 x 128 from 100 of those on; each with partial tiles in every dimension.
# Tolerance as above (64 iterations of FP32 products: 1e-5).
@pytest.mark.parametrize("m,n,B", [(33, 71, 35), (1290, 1301, 199), (1281, 1290, 1250)],
                         ids=["32x32", "64x32", "128x128"])
def test_shared_fp32_product_tiles_match_oracle(C, m, n, B):
    d = shared_dense_lp_batch(m, n, B, seed=m + B, bound_frac=0.5)
    opts = dict(eps_abs=1e-14, eps_rel=1e-14, iteration_limit=64, power_max_iter=0)
    h = C.mpax_lp_shared_create(m, n, B, d["A"], d["C"], d["b"], d["b"], d["l"], d["u"])
    try:
        C.mpax_shared_solve(h, C.mpax_options_default(fp64_continuation=0, **opts), True)
        X, Y = C.mpax_shared_get_solution(h, m, n, B)
    finally:
        C.mpax_shared_destroy(h)
    for k in (0, B // 2, B - 1):
        ref = O.solve_lp(_oracle_problem(d, k), O.Options(
            eps_primal_infeasible=0.0, eps_dual_infeasible=0.0, **opts))
        assert rel_inf(X[k], ref.x) <= 1e-5, k
        assert rel_inf(Y[k], ref.y) <= 1e-5, k


# The updates run blocks of whole warps, no wider than an instance has items: 1, 31 and 33
# items per thread group, four coordinates per thread (multiples of four) and one.
@pytest.mark.parametrize("m,n", [(3, 1), (4, 12), (8, 128), (31, 132), (33, 124), (132, 33)])
def test_shared_narrow_instances_match_oracle(C, m, n):
    B = 40
    d = shared_dense_lp_batch(m, n, B, seed=m * 7 + n, bound_frac=0.5)
    opts = dict(eps_abs=1e-14, eps_rel=1e-14, iteration_limit=64, power_max_iter=0)
    h = C.mpax_lp_shared_create(m, n, B, d["A"], d["C"], d["b"], d["b"], d["l"], d["u"])
    try:
        C.mpax_shared_solve(h, C.mpax_options_default(fp64_continuation=0, **opts), True)
        X, Y = C.mpax_shared_get_solution(h, m, n, B)
    finally:
        C.mpax_shared_destroy(h)
    for k in (0, B - 1):
        ref = O.solve_lp(_oracle_problem(d, k), O.Options(
            eps_primal_infeasible=0.0, eps_dual_infeasible=0.0, **opts))
        assert rel_inf(X[k], ref.x) <= 1e-5, k
        assert rel_inf(Y[k], ref.y) <= 1e-5, k


def test_shared_many_tiny_instances_gain_from_four_coordinates_a_thread(C):
    """20,000 instances of 12 columns (four coordinates per thread) take at most the ratio
    of the columns longer than those of 11 (one per thread)."""
    import time

    import torch
    best = {}
    for n in (11, 12):
        rng = np.random.default_rng(n)
        A = rng.standard_normal((8, n)).astype(np.float32)
        b = A.astype(np.float64) @ rng.random(n)
        h = C.mpax_lp_shared_create(8, n, 20000, A, rng.standard_normal((20000, n)), b, b,
                                    np.zeros(n), np.ones(n))
        opts = C.mpax_options_default(iteration_limit=640, eps_abs=1e-14, eps_rel=1e-14,
                                      power_max_iter=0, fp64_continuation=0)
        try:
            ts = []
            for _ in range(5):
                torch.cuda.synchronize()
                t = time.perf_counter()
                C.mpax_shared_solve(h, opts, True)
                torch.cuda.synchronize()
                ts.append(time.perf_counter() - t)
        finally:
            C.mpax_shared_destroy(h)
        best[n] = min(ts)
    assert best[12] <= best[11] * 12 / 11


def test_shared_very_many_instances_use_little_memory_and_the_same_weights(C):
    """262,144 instances of 3 x 5 take less than 1 KB each on the device, and their step
    weights, formed for 16 iterations at a time, give the bits of a small batch's, formed at
    once for the whole block."""
    import torch
    m, n, B, few = 3, 5, 1 << 18, 40
    d = shared_dense_lp_batch(m, n, B, seed=3, bound_frac=0.5)
    opts = C.mpax_options_default(iteration_limit=400, check_every=200, eps_abs=1e-14, eps_rel=1e-14,
                                  power_max_iter=0, fp64_continuation=0)
    X, Y = {}, {}
    for b in (few, B):
        before = torch.cuda.mem_get_info()[0]
        h = C.mpax_lp_shared_create(m, n, b, d["A"], np.ascontiguousarray(d["C"][:b]), d["b"], d["b"],
                                    d["l"], d["u"])
        try:
            if b == B:
                assert before - torch.cuda.mem_get_info()[0] < 1024 * B
            C.mpax_shared_solve(h, opts, True)
            X[b], Y[b] = C.mpax_shared_get_solution(h, m, n, b)
        finally:
            C.mpax_shared_destroy(h)
    np.testing.assert_array_equal(X[few], X[B][:few])
    np.testing.assert_array_equal(Y[few], Y[B][:few])
