"""Host threads that solve networks at the same time: small ones run their resident iterations on a half
of the SMs each, the others take turns. What each gets is bit for bit what it gets alone, whatever
its launches ran on: networks of one CTA, of up to half the SMs and of all, every storage type,
scalar tails in few and in many iterations, a fixed count and a stop test."""
import threading

import numpy as np
import pytest

from paper_2501_17996_gb300 import instances as I

pytestmark = pytest.mark.gpu


def _powij(n, seed):
    inst = I.ring_random_instance(n, 4, seed, "u1_10", "pow", gamma=0.5)
    inst.gamma = np.random.default_rng(seed).uniform(0.3, 0.7, size=(n, n))
    return inst


def _log(n, deg, seed):
    return I.ring_random_instance(n, deg, seed, "u1_10", "log")


FIXED = dict(stop_mode="none", max_iters=1500, k_check=50)
WORK = [
    (lambda: _log(5, 2, 0), FIXED),
    (lambda: _log(100, 10, 1), dict(FIXED, k_adapt=7)),
    (lambda: _log(100, 10, 2), dict(stop_mode="kkt", eps=1e-3, max_iters=4000, k_check=50)),
    (lambda: _log(300, 8, 3), FIXED),
    (lambda: _log(900, 8, 4), FIXED),
    (lambda: _log(200, 8, 5), dict(FIXED, precision="bf16")),
    (lambda: _powij(90, 6), dict(FIXED, precision="fp64", max_iters=300)),
    (lambda: I.ring_random_instance(260, 6, 7, "lognormal", "pow", gamma=0.4), FIXED),
    (lambda: _log(40, 4, 8), dict(FIXED, k_check=1)),
    (lambda: _log(110, 8, 9), dict(FIXED, precision="bf16")),
]


def test_solves_at_the_same_time_equal_solves_alone(lib):
    keys = ("iters", "rc", "omega", "rel_kkt", "utility", "dual_bound")
    probs = [lib.Problem(make()) for make, _ in WORK]

    def solve(i):
        return probs[i].solve(want_F=True, raise_on_error=False, **WORK[i][1])

    alone = [solve(i) for i in range(len(WORK))]
    for _ in range(3):
        got = [None] * len(WORK)
        start = threading.Barrier(len(WORK))

        def go(i):
            start.wait()
            got[i] = solve(i)

        threads = [threading.Thread(target=go, args=(i,)) for i in range(len(WORK))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for a, g in zip(alone, got):
            assert [g[k] for k in keys] == [a[k] for k in keys]
            assert np.array_equal(g["T"], a["T"]) and np.array_equal(g["F"], a["F"])
    for p in probs:
        p.close()
