"""What a re-solve uploads: after any order of weight and capacity changes, in the direct and the
batched path, a cold solve is bit-identical to that of a new problem with the same data."""
import numpy as np
import pytest

from paper_2501_17996_gb300 import instances as I

pytestmark = pytest.mark.gpu


def _with(inst, cap, w):
    return I.Instance(inst.n, inst.tail, inst.head, cap, inst.kind, w, inst.gamma)


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("order", ["c", "w", "cw", "wc", "cc"])
def test_cold_solve_after_updates_equals_a_new_problem(lib, order, batched):
    base = I.ring_random_instance(97, 4, 1, "u1_10", "pow", gamma=0.4)
    rng = np.random.default_rng(2)
    opts = lib.mcf_options_default(stop_mode="none", max_iters=20, k_check=10)

    def solve(p):
        if batched:
            return lib.mcf_solve_batch([p], opts, want_T=True)[1][0]["T"]
        return p.solve(stop_mode="none", max_iters=20, k_check=10)["T"]

    cap, w = base.cap, base.w
    with lib.Problem(base) as p:
        solve(p)
        for what in order:
            if what == "c":
                cap = rng.uniform(1.0, 10.0, cap.size)
                p.update_capacities(cap)
            else:
                w = rng.uniform(0.5, 1.5, w.shape)
                np.fill_diagonal(w, 0.0)
                p.update_weights(w)
            got = solve(p)
            with lib.Problem(_with(base, cap, w)) as fresh:
                assert np.array_equal(got, solve(fresh))
