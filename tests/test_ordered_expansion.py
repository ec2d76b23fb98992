"""Ordered expansion of FREE models: a state proposes a unit only when no
later unit has started, so every state is generated once and no visited set is
kept.

On the CPU the rule is restated and compared with the oracle's general search;
on the GPU the ordered pass is compared with the oracle, with a pass that uses
the visited set, and at sizes of many tiles with the closed forms."""
import pytest

import closed_forms as CF
import replay as RP
from paper_2305_09130_gb300 import workloads as W

NO_LIMIT = (1 << 64) - 1


def ordered_widths(spec, T, prune):
    """Level widths (levels 0..) of the ordered generation, checking that no
    state comes up twice."""
    level = [(k, (0,) * spec.P) for k in range(spec.a * spec.b)]
    widths = [1, spec.a, len(level)]
    while level:
        nxt = []
        for k, n in level:
            if sum(n) == spec.n_workgroups[k]:
                continue
            top = max((c for c in range(spec.P) if n[c]), default=0)
            for c in range(top, spec.P):
                m = n[:c] + (n[c] + 1,) + n[c + 1:]
                if not prune or max(x * s for x, s in zip(m, spec.speed)) * spec.cost[k] <= T:
                    nxt.append((k, m))
        assert len(nxt) == len(set(nxt))
        if nxt:
            widths.append(len(nxt))
        level = nxt
    return widths


@pytest.mark.parametrize("P", [1, 2, 3, 5, 8])
def test_ordered_generation_is_the_general_search(oracle, P):
    spec = W.random_small(6100 + P, P, 2, 2, 9 if P < 5 else 5, cost_max=6, speed_max=3)
    t_min = oracle.min_time(spec)["t_min"]
    for T in (0, t_min - 1, t_min, 2 * t_min, NO_LIMIT):
        for prune in (False, True):
            got = ordered_widths(spec, T, prune)
            exp = oracle.check(spec, T, prune=prune, early_exit=False, widths=max(spec.n_workgroups) + 3)
            assert got == exp["widths"] and sum(got) == exp["states"]


def gpu_models():
    """Every number of units, 64- and 128-bit keys, a long narrow model, clocks
    beyond 32 bits (keys of more than 64 used bits: below)."""
    out = []
    for P in range(1, 17):
        n_max = {1: 60, 2: 30, 3: 14, 4: 9}.get(P, 6 if P < 9 else 4)
        out.append(W.random_small(6200 + P, P, 2, 3, n_max, cost_max=6, speed_max=3, key_bits=128 if P % 2 else 0))
    long = W.ModelSpec("long_fields", 2, [1, 2], [1, 2], [300, 2, 3, 299], [2, 5, 3, 1], [1, 2], key_bits=128)
    out.append(long)
    big = W.random_small(6240, 3, 2, 2, 10, cost_max=5, speed_max=2)
    big.cost = [c + (1 << 31) for c in big.cost]
    out.append(big)
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("spec", gpu_models(), ids=lambda s: f"{s.name}_P{s.P}_k{s.key_bits}")
def test_ordered_pass_matches_oracle_and_visited_set(mc, oracle, spec):
    t_min = oracle.min_time(spec)["t_min"]
    opts = [{}, {"no_log_tags": 1}, {"threads_per_block": 64, "blocks_per_sm": 1}, {"probe_scheme": "split"}]
    models = [mc.mc_model_create(spec, mc.mc_options_default(engine="level", **o)) for o in opts]
    lay = mc.mc_model_layout(models[0])
    for m in models:
        assert mc.mc_count_states(m) == oracle.count(spec)
        assert mc.mc_last_widths(m) == CF.widths(spec)
    for T in (0, t_min - 1, t_min, t_min + 1, 2 * t_min, NO_LIMIT):
        for prune, ee in ((1, 1), (0, 1), (1, 0), (0, 0)):
            exp = oracle.check(spec, T, prune=bool(prune), early_exit=bool(ee))
            for m in models:
                mc.mc_set_options(m, mc.mc_options_default(engine="level", prune=prune, early_exit=ee))
                r = mc.mc_check(m, T)
                assert (r["holds"], r["states"], r["levels"]) == (exp["holds"], exp["states"], exp["levels"])
                if exp["holds"]:
                    continue
                i, j, n = RP.decode(lay, r["cex_key"])
                assert (r["cex_time"], i - 1, j - 1, r["cex_level"], n) == (
                    exp["cex_time"], exp["cex_i"], exp["cex_j"], exp["cex_level"], exp["cex_n"])
                assert r["trace"][-1] == r["cex_key"] and len(r["trace"]) == r["cex_level"] + 1
                RP.replay(spec, lay, r["trace"], lambda t: t <= T)
    for search in ("single", "lower", "bisect"):
        exp = oracle.min_time(spec, search=search)
        mc.mc_set_options(models[0], mc.mc_options_default(engine="level", search=search))
        r = mc.mc_min_time(models[0])
        for k in ("t_min", "t_ini", "states", "checks", "i", "j", "level"):
            assert r[k] == exp[k]
        RP.replay(spec, lay, r["trace"], lambda t: t == r["t_min"])


@pytest.mark.gpu
@pytest.mark.parametrize("spec", [W.c3(G=20, rule=W.FREE), W.c3(G=21, rule=W.FREE, key_bits=0), W.c2(G=61, rule=W.FREE),
                                  W.random_small(6301, 5, 3, 2, 45, speed_max=3),
                                  W.ModelSpec("used_62", 15, [1], [1], [8], [3], [1, 2, 2] * 5),
                                  W.ModelSpec("used_66", 16, [1], [1], [8], [3], [1, 2] * 8)], ids=lambda s: f"{s.name}_k{s.key_bits}")
def test_ordered_pass_over_many_tiles(mc, spec):
    """Levels of one key per thread, of several and of many tiles (up to
    millions of states), and keys computed in 128 bits, against the closed
    forms."""
    m = mc.mc_model_create(spec, mc.mc_options_default(engine="level"))
    assert mc.mc_count_states(m) == CF.count(spec)
    assert mc.mc_last_widths(m) == CF.widths(spec)
    t, _cfgs = CF.tmin(spec)
    for prune in (1, 0):
        mc.mc_set_options(m, mc.mc_options_default(engine="level", prune=prune))
        r = mc.mc_min_time(m)
        assert r["t_min"] == t
        RP.replay(spec, mc.mc_model_layout(m), r["trace"], lambda x: x == t)


@pytest.mark.gpu
@pytest.mark.parametrize("tags", [0, 1])
def test_ordered_pass_reports_a_full_log(mc, tags):
    m = mc.mc_model_create(W.c1(W.FREE), mc.mc_options_default(engine="level", log_capacity=100, no_log_tags=1 - tags))
    for _ in range(2):
        with pytest.raises(mc.MCError) as e:
            mc.mc_count_states(m)
        assert e.value.code == mc.MC_ERR_FRONTIER
