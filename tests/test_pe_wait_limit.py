"""PE-level model: mc_options.barrier_timeout_ns limits each device-wide wait,
not a search.  Narrow levels are explored by one block while the others wait,
so a search of any length has to pass under a limit far below its own time."""
import time

import pytest

from paper_2305_09130_gb300 import pe_workloads as PW
from test_pe_ordered import gpu_models

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tags", [0, 1])
def test_a_long_narrow_search_outlasts_the_wait_limit(mc, tags):
    ticks, rounds = 60_000, 2  # one PE: a mark and a tick per clock tick, one state per level
    spec = PW.PeSpec("long", 1, [1], [1], [rounds], [1], [[(ticks, 1)]])
    m = mc.mc_pe_model_create(spec, mc.mc_options_default(barrier_timeout_ns=20_000_000, no_log_tags=1 - tags))
    mc.mc_pe_count_states(m)  # (allocations)
    t0 = time.perf_counter()
    assert mc.mc_pe_count_states(m) == 3 + rounds * (1 + 2 * ticks)
    assert time.perf_counter() - t0 > 5 * 0.02  # the limit was passed many times over
    assert mc.mc_pe_last_widths(m, cap=1 << 20) == [1] * (3 + rounds * (1 + 2 * ticks))
    r = mc.mc_pe_min_time(m)
    assert r["t_min"] == rounds * ticks and len(r["trace"]) == 3 + rounds * (1 + 2 * ticks)


@pytest.mark.parametrize("spec", gpu_models(), ids=lambda s: f"{s.name}_P{s.P}")
def test_a_short_wait_limit_changes_no_answer(mc, spec):
    """Block 0 then leaves the narrow levels every half millisecond, at widths
    below and above the one at which it takes them over."""
    answers = []
    for limit in (0, 2_000_000):
        m = mc.mc_pe_model_create(spec, mc.mc_options_default(barrier_timeout_ns=limit))
        count = mc.mc_pe_count_states(m)
        r = mc.mc_pe_min_time(m)
        answers.append((count, mc.mc_pe_last_widths(m), {k: v for k, v in r.items() if k != "trace"}, len(r["trace"])))
    assert answers[0] == answers[1]
