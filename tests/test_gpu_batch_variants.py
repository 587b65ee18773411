"""The batched phases at the edges of their variants: rows that fill a warp's chunks exactly and
one entry more (1, 2, 4 and 8 chunks per lane, and the first longer shape), instances smaller than
a run, nodes with more than 32 incident edges, sums in every iteration and only in some, exponents
of 1/2 among others, forced shapes; all in one batch against the FP64 oracle.

Tolerance: FP32 rounding (6e-8) through at most 10 iterations of sums of at most 40 terms leaves
below 1e-5 of the largest entry; 1e-4 as in the batch trajectory test."""
import numpy as np
import pytest

from oracle import pdmcf as O
from paper_2501_17996_gb300 import instances as I

pytestmark = pytest.mark.gpu

TOL = 1e-4


def _dense(n, seed):
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


def _mix():
    r = I.ring_random_instance
    return [r(3, 1, 0, "u1_10", "log"), r(128, 4, 1, "u1_10", "log"), r(129, 3, 2, "u1_10", "log"),
            r(256, 3, 3, "lognormal", "pow", gamma=0.4), r(257, 3, 4, "u1_10", "log"), _dense(60, 5),
            r(512, 2, 6, "lognormal", "pow", gamma=0.5), r(513, 2, 7, "u1_10", "log"), _powij(65, 8),
            r(1024, 2, 9, "u1_10", "log"), r(1025, 2, 10, "u1_10", "log")]


def _small():
    return [I.ring_random_instance(40 + 8 * i, 3, i, "u1_10", "log") for i in range(5)]


@pytest.mark.parametrize("make,iters,k_check,k_adapt,shape", [
    (_mix, 8, 4, 1, -1), (_mix, 7, 7, 100, -1), (_small, 10, 3, 4, 3), (_small, 10, 10, 3, 5)])
def test_batch_variants_match_oracle(lib, make, iters, k_check, k_adapt, shape):
    insts = make()
    probs = [lib.Problem(i) for i in insts]
    opts = lib.mcf_options_default(stop_mode="none", max_iters=iters, k_check=k_check, k_adapt=k_adapt,
                                   shape=shape)
    _, res = lib.mcf_solve_batch(probs, opts, want_T=True, want_Y=True)
    for inst, g in zip(insts, res):
        ref = O.pdmcf(inst.n, inst.tail, inst.head, inst.cap, inst.kind, inst.w, inst.gamma,
                      stop_mode="none", max_iters=iters, k_check=k_check, k_adapt=k_adapt)
        off = ~np.eye(inst.n, dtype=bool)
        assert g["iters"] == iters
        assert np.abs(g["T"][off] - ref.T[off]).max() <= TOL * np.abs(ref.T[off]).max()
        assert np.abs(g["Y"][off] - ref.Yhat[off]).max() <= TOL * np.abs(ref.Yhat[off]).max()
        assert g["omega"] == pytest.approx(ref.omega, rel=TOL)
    for p in probs:
        p.close()
