"""Solves of several handles at the same time, from threads of one process."""
import threading
import time

import numpy as np
import pytest

from synth import instance_seed, lp_instance, ragged_lp_batch
from tests.gpu_util import create, lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    return lib()


def test_a_solve_beside_a_batch_that_keeps_half_of_the_gpu(C):
    """No kernel of a single solve needs the whole GPU at once: beside a ragged batch that
    keeps half of the SMs for a second or more, solves end before the batch does."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    d = ragged_lp_batch(sms // 2, seed=3, m_lo=4000, m_hi=4200, density=0.004)
    hb = C.mpax_lp_batch_create(d["B"], *[d[k] for k in ("m_off", "n_off", "row_ptr", "col", "val",
                                                        "c", "lc", "uc", "l", "u")])
    lp = lp_instance(6000, 9000, seed=instance_seed(303), density=0.003)
    h = create(C, lp)
    opts = C.mpax_options_default(iteration_limit=64, eps_abs=1e-14, eps_rel=1e-14)
    C.mpax_solve(h, opts)
    x0, y0 = C.mpax_get_solution(h, lp["m"], lp["n"])
    ended = []
    batch = threading.Thread(target=lambda: (C.mpax_batch_solve(hb, C.mpax_options_default(
        eps_abs=1e-14, eps_rel=1e-14, power_max_iter=0, iteration_limit=100000, time_limit=3.0)),
        ended.append(time.perf_counter())))
    try:
        batch.start()
        time.sleep(0.3)
        solved = []
        for _ in range(3):
            C.mpax_solve(h, opts)
            solved.append(time.perf_counter())
        batch.join()
        x, y = C.mpax_get_solution(h, lp["m"], lp["n"])
    finally:
        C.mpax_destroy(h)
        C.mpax_batch_destroy(hb)
    assert solved[-1] < ended[0]
    np.testing.assert_array_equal(x, x0)
    np.testing.assert_array_equal(y, y0)


def test_four_threads_solve_as_one_after_another(C):
    """LPs of four threads, each on its own handle, give the bits that they give alone."""
    lps = [lp_instance(3000 + 500 * i, 5000, seed=instance_seed(400 + i), density=0.003)
           for i in range(4)]
    opts = C.mpax_options_default(iteration_limit=640, eps_abs=1e-14, eps_rel=1e-14)
    hs = [create(C, d) for d in lps]
    try:
        alone = []
        for h, d in zip(hs, lps):
            C.mpax_solve(h, opts)
            alone.append(C.mpax_get_solution(h, d["m"], d["n"]))
        threads = [threading.Thread(target=lambda h=h: [C.mpax_solve(h, opts) for _ in range(5)])
                   for h in hs]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for h, d, (x, y) in zip(hs, lps, alone):
            got = C.mpax_get_solution(h, d["m"], d["n"])
            np.testing.assert_array_equal(got[0], x)
            np.testing.assert_array_equal(got[1], y)
    finally:
        for h in hs:
            C.mpax_destroy(h)
