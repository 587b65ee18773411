"""BF16-stored flows: the automatic choice of kernels gives the bits of the per-phase kernels of the
same shape (which a timed solve launches). Roundings of F to BF16 amplify a last-place difference
of Y or of a multiplier to 2^-8 of an entry, so a route that only agrees to FP32 rounding changes
the outputs visibly. Sizes on both sides of the lines between the routes: rows of the resident
iteration, of the register shapes (1025 to 2047 entries) and of the in-sum kind, renumbered
networks, each utility."""
import numpy as np
import pytest

from paper_2501_17996_gb300 import instances as I

pytestmark = pytest.mark.gpu

CASES = [
    lambda: I.ring_random_instance(300, 4, 7, "lognormal", "pow", gamma=0.5),
    lambda: I.ring_random_instance(1025, 3, 9, "lognormal", "pow", gamma=0.5),
    lambda: I.ring_random_instance(2047, 3, 9, "lognormal", "pow", gamma=0.4),
    lambda: I.ring_random_instance(2049, 5, 9, "lognormal", "pow", gamma=0.5),
    lambda: I.ring_random_instance(3001, 4, 11, "lognormal", "pow", gamma=0.5),
    lambda: I.ring_random_instance(1025, 3, 9, "u1_10", "log"),
    lambda: I.ring_random_instance(2040, 4, 10, "u1_10", "log"),
    lambda: I.ring_random_instance(2049, 5, 10, "u1_10", "log"),
    lambda: I.ring_random_instance(3001, 4, 12, "u1_10", "log"),
    lambda: I.knn(1500, 6, 3),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_automatic_route_keeps_the_bits(lib, case):
    inst = CASES[case]()
    opts = dict(precision="bf16", stop_mode="none", max_iters=25, k_check=10, k_adapt=7)
    with lib.Problem(inst) as p:
        a = p.solve(want_T=True, **opts)
        b, _ = p.solve_timed(want_T=True, **opts)
    assert a["iters"] == b["iters"] == 25
    assert np.array_equal(a["T"], b["T"])
    assert a["utility"] == b["utility"] and a["dual_bound"] == b["dual_bound"] and a["omega"] == b["omega"]
