"""The stop rule that the resident iteration evaluates on the device, against the rule written out here
and read over the solve's own check log: the measure's target, the paper's residual, the rounding
floor (stall_checks, with the restart when omega stops adapting), the hand-over of BF16-stored flows
to the FP32 polish, and the iteration cap. Each is solved without a log too (then the device decides
over up to 1000 iterations before the host looks) and must end the same; and with a register shape
other than the automatic one, whose rule the host evaluates."""
import json
import math

import numpy as np
import pytest

from paper_2501_17996_gb300 import instances as I

pytestmark = pytest.mark.gpu


def _replay(lines, mode, eps, stall_checks=0, handoff=0.0, handoff_stall=0):
    """(checks until the rule ends the solve, why); why is None if it never does."""
    floor, since, frozen, best, no_better = math.inf, 0, False, math.inf, 0
    for i, c in enumerate(lines):
        kkt = math.inf if c["rel_kkt"] is None else c["rel_kkt"]
        r = math.inf if c["r_over_nm"] is None else c["r_over_nm"]
        if (mode == "paper" and r < eps) or (mode == "kkt" and kkt < eps):
            return i + 1, "converged"
        if kkt < handoff:
            return i + 1, "handoff"
        if mode == "kkt" and stall_checks > 0 and kkt < 100.0 * eps:
            if frozen != (not c["omega_adapting"]):
                frozen, floor, since = not c["omega_adapting"], math.inf, 0
            if kkt < 0.95 * floor:
                floor, since = kkt, 0
            else:
                since += 1
                if since >= stall_checks:
                    return i + 1, "stalled"
        if handoff_stall > 0:
            if kkt < 0.95 * best:
                best, no_better = kkt, 0
            else:
                no_better += 1
                if no_better >= handoff_stall:
                    return i + 1, "handoff"
    return len(lines), None


def _other_shape(lib, p, **opts):
    auto = p.solve_timed(**{**opts, "max_iters": 1})[0]["shape"]
    chunks = ((p.n + 7) // 8 * 8) // (2 if opts.get("precision") == "fp64" else 4)
    return next(s for s, (g, v, _, kind) in enumerate(lib.mcf_shape_info())
                if kind == 0 and s != auto and g * v >= chunks)


CASES = [   # options, what ends the solve
    (dict(stop_mode="kkt", eps=1e-4, max_iters=20000, k_check=50), "converged"),
    (dict(stop_mode="kkt", eps=1e-6, max_iters=20000, k_check=30, precision="fp64"), "converged"),
    (dict(stop_mode="paper", eps=1e-3 / (100 * 99), max_iters=20000, k_check=7), None),
    (dict(stop_mode="kkt", eps=2e-6, max_iters=20000, k_check=10, stall_checks=4, compensated_duals=0), "stalled"),
    (dict(stop_mode="kkt", eps=1e-12, max_iters=1234, k_check=50), "cap"),
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("route", ["automatic", "host"])
def test_stop_rule_over_the_check_log(lib, tmp_path, case, route):
    opts, want = CASES[case]
    with lib.Problem(I.mid(1)) as p:
        if route == "host":
            opts = dict(opts, shape=_other_shape(lib, p, **opts))
        log = tmp_path / "log.jsonl"
        a = p.solve(check_log=str(log), raise_on_error=False, **opts)
        b = p.solve(raise_on_error=False, **opts)
    lines = [json.loads(x) for x in log.read_text().splitlines()]
    checks, why = _replay(lines, opts["stop_mode"], opts["eps"], opts.get("stall_checks", 100))
    assert checks == len(lines)                       # nothing ran past the rule
    assert a["iters"] == lines[-1]["k"]
    assert a["stalled"] == (why == "stalled")
    if why is None:
        assert a["iters"] == opts["max_iters"]
    assert a["rc"] == (lib.MCF_OK if why == "converged" else lib.MCF_ERR_NOT_CONVERGED)
    if want is not None:
        assert (why or "cap") == want
    assert (b["rc"], b["iters"], b["stalled"], b["rel_kkt"], b["omega"]) == \
           (a["rc"], a["iters"], a["stalled"], a["rel_kkt"], a["omega"])
    assert np.array_equal(a["T"], b["T"])
    if case == 0:
        assert a["iters"] > 1000                      # more than one group of launches


@pytest.mark.parametrize("eps", [1e-4, 1e-3])
def test_bf16_hand_over_follows_the_rule(lib, tmp_path, eps):
    """Log utility, so that the BF16 phase is resident too: within 10 eps of the target, or five
    checks without a 5 % improvement."""
    opts = dict(precision="bf16", stop_mode="kkt", eps=eps, max_iters=20000, polish_iters=20000, k_check=25)
    log = tmp_path / "log.jsonl"
    with lib.Problem(I.mid(1)) as p:
        a = p.solve(check_log=str(log), raise_on_error=False, **opts)
        b = p.solve(raise_on_error=False, **opts)
    lines = [json.loads(x) for x in log.read_text().splitlines()]
    first = [c for c in lines if c["precision"] == "bf16"]
    then = [c for c in lines if c["precision"] == "fp32"]
    checks, why = _replay(first, "kkt", eps, 100, handoff=10.0 * eps, handoff_stall=5)
    assert checks == len(first) and why in ("handoff", "converged", "stalled")
    if then:
        checks, why = _replay(then, "kkt", eps, 100)
        assert checks == len(then)
    assert a["iters"] == first[-1]["k"] + (then[-1]["k"] if then else 0)
    assert (b["rc"], b["iters"], b["rel_kkt"]) == (a["rc"], a["iters"], a["rel_kkt"])
    assert np.array_equal(a["T"], b["T"])
