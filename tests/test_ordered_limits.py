"""Ordered expansion of FREE models at the limits of its arithmetic: clocks
that exceed 32 bits by a unit's speed alone, and keys that fill their word,
compared with the oracle and with the pass that keeps a visited set; and a
probe limit set on a model that keeps none so far."""
import pytest

import replay as RP
from paper_2305_09130_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NO_LIMIT = (1 << 64) - 1
BIG = 1 << 31


def fast_and_slow(speed, n, cost):
    k = len(n)
    return W.ModelSpec("speeds_" + "_".join(map(str, speed)), len(speed), [1], list(range(1, k + 1)), n, cost, speed)


@pytest.mark.parametrize("spec", [fast_and_slow([BIG], [4, 3], [1, 2]),
                                  fast_and_slow([1, 2 * BIG - 1], [5, 2, 9], [3, 1, 2]),
                                  fast_and_slow([2 * BIG - 1, 1], [6, 3], [1, 4]),
                                  fast_and_slow([2 * BIG - 1, 2 * BIG - 1], [3, 5], [1, 1]),
                                  fast_and_slow([BIG, 7, BIG + 5], [4, 6], [2, 1]),
                                  fast_and_slow([1 << 30, BIG - 1, BIG, 3, BIG + 1], [5, 4], [1, 1])],
                         ids=lambda s: s.name)
def test_speeds_beyond_32_bits_of_clock(mc, oracle, spec):
    t_min = oracle.min_time(spec)["t_min"]
    models = [mc.mc_model_create(spec, mc.mc_options_default(engine="level", **o)) for o in ({}, {"probe_scheme": "split"})]
    lay = mc.mc_model_layout(models[0])
    for T in (0, t_min - 1, t_min, (1 << 32) - 1, 1 << 32, 3 * BIG, 1 << 33, 1 << 34, NO_LIMIT):
        for prune, ee in ((1, 1), (0, 1), (1, 0), (0, 0)):
            exp = oracle.check(spec, T, prune=bool(prune), early_exit=bool(ee))
            for m in models:
                mc.mc_set_options(m, mc.mc_options_default(engine="level", prune=prune, early_exit=ee))
                r = mc.mc_check(m, T)
                assert (r["holds"], r["states"], r["levels"]) == (exp["holds"], exp["states"], exp["levels"])
                if not exp["holds"]:
                    i, j, n = RP.decode(lay, r["cex_key"])
                    assert (r["cex_time"], i - 1, j - 1, r["cex_level"], n) == (
                        exp["cex_time"], exp["cex_i"], exp["cex_j"], exp["cex_level"], exp["cex_n"])
                    RP.replay(spec, lay, r["trace"], lambda t: t == r["cex_time"])
    for search in ("single", "lower", "bisect"):
        exp = oracle.min_time(spec, search=search)
        for m in models:
            mc.mc_set_options(m, mc.mc_options_default(engine="level", search=search))
            r = mc.mc_min_time(m)
            assert {k: r[k] for k in ("t_min", "t_ini", "states", "checks", "i", "j", "level")} == {
                k: exp[k] for k in ("t_min", "t_ini", "states", "checks", "i", "j", "level")}


def test_keys_that_fill_their_word(mc):
    """64 used bits leave no room for a tag, and the upper half of a key is all
    ones in the last configuration (1023, 511) from n_0 = 32764 on.  Pruning
    keeps the other configurations and units from starting."""
    a, b, N = 1023, 511, 32767
    spec = W.ModelSpec("ones", 3, list(range(a)), list(range(b)), [1] * (a * b - 1) + [N],
                       [N + 1] * (a * b - 1) + [1], [1, N + 1, N + 1])
    got = []
    for o in ({}, {"table_log2": 20}):
        m = mc.mc_model_create(spec, mc.mc_options_default(engine="level", log_capacity=600_000,
                                                           barrier_timeout_ns=2_000_000_000, **o))
        lay = mc.mc_model_layout(m)
        assert lay["used_bits"] == 64 and lay["log_tag_bits"] == 0
        r = mc.mc_check(m, N)
        assert r["cex_key"] >> 32 == 0xFFFFFFFF
        assert (r["cex_time"], r["cex_i"], r["cex_j"], r["cex_level"]) == (N, a - 1, b - 1, 2 + N)
        assert r["states"] == 1 + a + a * b + N
        RP.replay(spec, lay, r["trace"], lambda t: t == N)
        got.append({k: v for k, v in r.items() if k != "trace"})
        mc.mc_model_destroy(m)
    assert got[0] == got[1]


@pytest.mark.parametrize("allocator", ["torch", None])
def test_a_probe_limit_set_later_acts(mc, allocator):
    """mc_options.max_probes acts on later queries, also of a model that was
    laid out without a visited set: one bucket probe cannot place the wide
    levels of 737,855 states, 64 can."""
    spec = W.c2(G=40, rule=W.FREE)
    m = mc.mc_model_create(spec, mc.mc_options_default(engine="level"), allocator=allocator)
    small = mc.mc_model_layout(m)["device_bytes"]
    exp = mc.mc_min_time(m, trace=False)
    assert mc.mc_count_states(m) == 737_855
    widths = mc.mc_last_widths(m)
    for limit in (1, 64, 1, 0):
        mc.mc_set_options(m, mc.mc_options_default(engine="level", max_probes=limit))
        if limit == 1:
            with pytest.raises(mc.MCError) as e:
                mc.mc_count_states(m)
            assert e.value.code == mc.MC_ERR_TABLE_FULL
            assert mc.mc_model_layout(m)["device_bytes"] > small
            continue
        assert mc.mc_count_states(m) == 737_855 and mc.mc_last_widths(m) == widths
        assert mc.mc_min_time(m, trace=False) == exp
    mc.mc_model_destroy(m)
