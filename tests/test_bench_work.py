"""The work figures of a bench line describe the launch that was timed: where the
timed kernel has no counters, the counts of a solve with counters (another kernel)
are left out.  The rule is the library's own (use_guided in eik_api.cu)."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

ST = {"evals": 100, "decreases": 70, "good": 10, "visits": 5, "pushes": 6, "stale_pops": 1, "rounds": 40,
      "solve_ms": 1.0}
AUTOTUNED = {"delta": 0.0, "k_delta": 0.375, "capacity": 4096, "ctas_per_sm": 20, "window": 31, "band": 6.0,
             "arith": 3, "tile": 1}


@pytest.mark.parametrize("opts", [{}, {"arith": 3, "tile": 2, "k_delta": 4.0}, {"capacity": 16}, {"timeout_ms": 5},
                                  {"sched_flags": 1 << 6}, AUTOTUNED, {"tile": 0, "delta": 0.0}])
def test_kernels_without_counters(opts):
    w = bench.work_per_step(ST, opts)
    assert w["good"] == 10 and w["note"]
    assert all(w[k] is None for k in ("evals", "decreases", "visits", "pushes", "stale_pops", "rounds", "empty", "bad"))


@pytest.mark.parametrize("opts", [{"arith": 1}, {"arith": 2}, {"tile": 1}, {"k_delta": 2.0}, {"window": 4},
                                  {"ctas_per_sm": 2}, {"band": 1.0}, {"delta": 0.1}, {"update": 2},
                                  {"update": 1, "arith": 3}, {"sched_flags": 1}, {"sched_flags": 2, "arith": 3},
                                  dict(AUTOTUNED, arith=1)])
def test_kernel_with_counters(opts):
    w = bench.work_per_step(ST, opts)
    assert "note" not in w and w["evals"] == 100 and w["empty"] == 30 and w["bad"] == 60 and w["rounds"] == 40
