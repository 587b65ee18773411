"""The resident iteration's grid barrier gives up after a bounded number of polls, once per solve:
with an arrival that never comes (mcf_test_withhold_next_arrival) the solve reports MCF_ERR_CUDA
after one wait, although some forty launches are queued behind the one that gave up, and the next
solve on the same problem is right. Long chunks are cut into launches of at most 1000 iterations,
with the same results."""
import time

import numpy as np
import pytest

from paper_2501_17996_gb300 import instances as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k_adapt", [(10, 100), (200, 2)])   # few and all SMs; 40 and 1000 launches
def test_barrier_gives_up_once_and_the_next_solve_is_right(lib, n, k_adapt):
    inst = I.ring_random_instance(n, 4, 0, "u1_10", "log")
    opts = dict(stop_mode="none", max_iters=1000, k_check=50, k_adapt=k_adapt)
    with lib.Problem(inst) as p, lib.Problem(inst) as other:
        ref = other.solve(want_T=True, **opts)
        lib.mcf_test_withhold_next_arrival()
        t0 = time.perf_counter()
        with pytest.raises(lib.MCFError) as ei:
            p.solve(**opts)
        waited = time.perf_counter() - t0
        assert ei.value.code == lib.MCF_ERR_CUDA
        assert "bounded device-side wait" in lib.mcf_last_error()
        print(f"gave up after {waited:.2f} s")
        assert waited < 10.0, waited           # one wait; forty of them would be a minute
        r = p.solve(want_T=True, warm_start=1, **opts)   # the iterate is invalid: starts cold
        assert r["iters"] == 1000 and np.array_equal(r["T"], ref["T"])


def test_long_chunks_are_cut_into_launches(lib):
    """2500 iterations without a scalar tail between the first and the last: three launches of the
    plain kernel, against chunks of 250 (k_adapt beyond the run, so both take the same steps). A wrong
    split (parity, barrier count) is an error of order one; rounding over 2500 contracting
    iterations stays far below 1e-3 of the largest entry."""
    inst = I.ring_random_instance(40, 4, 1, "u1_10", "log")
    with lib.Problem(inst) as p:
        a = p.solve(want_T=True, stop_mode="none", max_iters=2500, k_check=2500, k_adapt=10**6)
        b = p.solve(want_T=True, stop_mode="none", max_iters=2500, k_check=250, k_adapt=10**6)
    assert a["iters"] == b["iters"] == 2500
    assert np.abs(a["T"] - b["T"]).max() <= 1e-3 * np.abs(b["T"]).max()
    assert a["omega"] == pytest.approx(b["omega"], rel=1e-6)
