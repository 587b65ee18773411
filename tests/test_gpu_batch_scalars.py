"""The batched engine's scalar tail decides per iteration whether the sums are needed (a multiple
of k_adapt, or a stop test) from scalars that the same block then moves on. Every pattern of
summed and skipped iterations in turn, against the oracle: each iteration summed, every second and
third, and stop tests between them, so that a decision read after the move would show in omega."""
import numpy as np
import pytest

from oracle import pdmcf as O
from paper_2501_17996_gb300 import instances as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k_adapt,k_check", [(1, 7), (2, 9), (3, 5), (4, 1), (100, 3)])
def test_summed_and_skipped_iterations_match_the_oracle(lib, k_adapt, k_check):
    insts = [I.ring_random_instance(n, 4, n, "u1_10", "log") for n in (12, 33, 130, 200)]
    ref = [O.pdmcf(i.n, i.tail, i.head, i.cap, i.kind, i.w, i.gamma, stop_mode="none", max_iters=31,
                   k_check=k_check, k_adapt=k_adapt) for i in insts]
    opts = lib.mcf_options_default(stop_mode="none", max_iters=31, k_check=k_check, k_adapt=k_adapt)
    ps = [lib.Problem(i) for i in insts]
    _, got = lib.mcf_solve_batch(ps, opts, want_T=True)
    for i, r, g in zip(insts, ref, got):
        off = ~np.eye(i.n, dtype=bool)
        assert g["iters"] == 31
        assert g["omega"] == pytest.approx(r.omega, rel=1e-4)
        assert np.abs(g["T"][off] - r.T[off]).max() <= 1e-4 * np.abs(r.T[off]).max()
    for p in ps:
        p.close()
