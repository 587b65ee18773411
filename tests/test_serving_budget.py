"""Admission counts the bytes that a slot takes: the problem's state and the engine's sums, which are
one FP64 set (seven fields) per 128-entry piece of a node's column and five per edge. A request of
exactly the budget is queued, one byte less refuses it. Admission is paused, so nothing runs; with
or without a GPU."""
import pytest

from paper_2501_17996_gb300 import instances as I


@pytest.mark.parametrize("n", [40, 128, 129, 1000])
def test_budget_counts_what_a_slot_takes(lib, n):
    with lib.Problem(I.ring_random_instance(n, 3, n, "u1_10", "log")) as p:
        pieces = ((n + 7) // 8 * 8 + 127) // 128
        need = p.device_bytes("fp32") + 8 * (5 * p.m + 7 * n * pieces)
        try:
            lib.mcf_serving_config(need - 1, 0)
            with pytest.raises(lib.MCFError) as ei:
                p.submit(precision="fp32")
            assert ei.value.code == lib.MCF_ERR_OOM_BUDGET
            lib.mcf_serving_config(need, 0)
            t = p.submit(precision="fp32")
            lib.mcf_cancel(t)
            assert lib.mcf_wait(t, 1000)["status"] == lib.MCF_ERR_CANCELLED
        finally:
            lib.mcf_serving_shutdown()
            lib.mcf_serving_config(120 * 10**9, 256)
