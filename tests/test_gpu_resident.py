"""The resident iteration (many iterations per launch, automatic shapes with short rows) and the
flat node phase (longer rows) against the oracle, at the edges of their variants: rows that fill a warp's chunks exactly and one entry
more, a network served by one CTA, nodes with more than 32 incident edges, a scalar tail in
every iteration, chunks that do not divide the iteration count, exponents of 1/2 among others;
and its stop test on the device against the driver's."""
import numpy as np
import pytest

from oracle import pdmcf as O
from paper_2501_17996_gb300 import instances as I

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-4, "fp64": 1e-8, "bf16": 3e-2}   # of the largest entry, as the trajectory tests


def _dense(n, seed):
    """Every node within 20 steps is a neighbour: in- and out-degree 20, 40 incident edges."""
    rng = np.random.default_rng(seed)
    t = np.repeat(np.arange(n), 20)
    h = (t + np.tile(np.arange(1, 21), n)) % n
    w = rng.uniform(0.5, 1.5, size=(n, n))
    np.fill_diagonal(w, 0.0)
    return I.Instance(n, t.astype(np.int32), h.astype(np.int32), rng.uniform(1.0, 10.0, t.size), "log", w)


def _powij(n, seed):
    inst = I.ring_random_instance(n, 4, seed, "u1_10", "pow", gamma=0.5)
    g = np.random.default_rng(seed).uniform(0.3, 0.7, size=(n, n))
    g[::3] = 0.5
    inst.gamma = g
    return inst


CASES = [   # (network, precision, iterations, k_check, k_adapt)
    (lambda: I.ring_random_instance(5, 2, 0, "u1_10", "log"), "fp32", 21, 10, 100),
    (lambda: I.ring_random_instance(128, 4, 1, "u1_10", "log"), "fp32", 17, 8, 5),
    (lambda: I.ring_random_instance(129, 4, 1, "u1_10", "log"), "fp32", 17, 8, 5),
    (lambda: I.ring_random_instance(257, 3, 2, "lognormal", "pow", gamma=0.4), "fp32", 12, 50, 1),
    (lambda: I.ring_random_instance(513, 3, 2, "lognormal", "pow", gamma=0.5), "fp32", 9, 4, 100),
    (lambda: I.ring_random_instance(1024, 3, 3, "u1_10", "log"), "fp32", 6, 3, 2),
    (lambda: _dense(60, 4), "fp32", 20, 7, 100),
    (lambda: _dense(60, 4), "fp64", 20, 7, 3),
    (lambda: _powij(65, 5), "fp64", 25, 10, 100),
    (lambda: _powij(70, 5), "fp32", 25, 10, 100),
    (lambda: I.ring_random_instance(511, 3, 6, "u1_10", "log"), "fp64", 6, 3, 100),
    (lambda: I.ring_random_instance(300, 4, 7, "u1_10", "log"), "bf16", 6, 3, 100),
    (lambda: I.ring_random_instance(513, 3, 8, "lognormal", "pow", gamma=0.4), "fp64", 8, 4, 100),
    (lambda: I.ring_random_instance(1025, 3, 9, "u1_10", "log"), "fp32", 7, 5, 100),
    (lambda: I.ring_random_instance(1025, 3, 9, "lognormal", "pow", gamma=0.5), "bf16", 6, 4, 3),
    (lambda: I.ring_random_instance(2051, 3, 10, "lognormal", "pow", gamma=0.6), "fp32", 5, 5, 100),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_resident_trajectory_matches_oracle(lib, case):
    make, precision, iters, k_check, k_adapt = CASES[case]
    inst = make()
    ref = O.pdmcf(inst.n, inst.tail, inst.head, inst.cap, inst.kind, inst.w, inst.gamma,
                  stop_mode="none", max_iters=iters, k_check=k_check, k_adapt=k_adapt)
    with lib.Problem(inst) as p:
        g = p.solve(precision=precision, stop_mode="none", max_iters=iters, k_check=k_check,
                    k_adapt=k_adapt, want_F=True, want_Y=True)
    off = ~np.eye(inst.n, dtype=bool)
    tol = TOL[precision]
    assert g["iters"] == iters
    assert np.abs(g["T"][off] - ref.T[off]).max() <= tol * np.abs(ref.T[off]).max()
    assert np.abs(g["Y"][off] - ref.Yhat[off]).max() <= tol * np.abs(ref.Yhat[off]).max()
    assert np.abs(g["F"] - ref.Fhat).max() <= tol * np.abs(ref.Fhat).max()
    assert g["omega"] == pytest.approx(ref.omega, rel=tol)
    assert np.all(np.diag(g["Y"]) == 0)


def test_stop_test_on_the_device_equals_the_driver(lib, tmp_path):
    """With a check log every chunk returns to the driver; without one the device decides."""
    inst = I.mid(1)
    with lib.Problem(inst) as p:
        a = p.solve(stop_mode="kkt", eps=1e-4)
        b = p.solve(stop_mode="kkt", eps=1e-4, check_log=str(tmp_path / "log.jsonl"))
        c = p.solve(stop_mode="kkt", eps=1e-4, max_iters=a["iters"] - 50)   # the check before
    assert a["rc"] == b["rc"] == lib.MCF_OK and a["iters"] == b["iters"]
    assert np.array_equal(a["T"], b["T"]) and a["rel_kkt"] == b["rel_kkt"]
    assert c["rc"] == lib.MCF_ERR_NOT_CONVERGED and c["iters"] == a["iters"] - 50
