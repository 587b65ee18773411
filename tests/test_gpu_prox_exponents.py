"""Power utility with exponents near 0 and 1 in the resident iteration (n = 65), the flat node phase
(n = 1100) and the batched engine, against the oracle. FP64: rounding (1.1e-16) through 25
iterations of sums of at most ten terms, amplified by 1/(1 - gamma) <= 20 in the traffic, is below
1e-12 of the largest entry; 1e-10 leaves room for the duals' scale. FP32 as the trajectory tests."""
import numpy as np
import pytest

from oracle import pdmcf as O
from paper_2501_17996_gb300 import instances as I

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-10, "fp32": 1e-4, "batch": 1e-4}


@pytest.mark.parametrize("gamma", [0.05, 0.1, 0.9, 0.95])
@pytest.mark.parametrize("n,iters,how", [(65, 25, "fp64"), (65, 25, "fp32"), (65, 25, "batch"), (1100, 5, "fp32")])
def test_exponents_near_the_ends(lib, gamma, n, iters, how):
    inst = I.ring_random_instance(n, 4, 5, "u1_10", "pow", gamma=gamma)
    opts = dict(stop_mode="none", max_iters=iters, k_check=10)
    ref = O.pdmcf(inst.n, inst.tail, inst.head, inst.cap, inst.kind, inst.w, inst.gamma, **opts)
    with lib.Problem(inst) as p:
        if how == "batch":
            g = lib.mcf_solve_batch([p], lib.mcf_options_default(**opts), want_T=True, want_Y=True)[1][0]
        else:
            g = p.solve(precision=how, want_Y=True, **opts)
    off = ~np.eye(n, dtype=bool)
    for got, want in ((g["T"], ref.T), (g["Y"], ref.Yhat)):
        assert np.abs(got[off] - want[off]).max() <= TOL[how] * np.abs(want[off]).max()
