"""Configuration engine: passes with a warp for every configuration, and with
more configurations (or segments) than warps, where each warp takes several
and counts them itself, against the oracle."""
import pytest

from paper_2305_09130_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def many(P, side, n_max, rule, seed):
    s = W.random_small(seed, P, side, side, n_max, rule=rule)
    s.wg_values = s.ts_values = list(range(1, side + 1))
    return s


@pytest.mark.parametrize("spec,opts", [(many(3, 120, 3, W.GREEDY, 71), {}), (many(10, 101, 2, W.GREEDY, 72), {}),
                                       (many(1, 150, 2, W.FREE, 73), {}), (many(2, 20, 3, W.GREEDY, 74), {"blocks_per_sm": 1}),
                                       (many(6, 30, 4, W.GREEDY, 75), {"blocks_per_sm": 1}),
                                       (W.random_small(76, 4, 2, 2, 3000, rule=W.GREEDY), {})],
                         ids=lambda x: f"P{x.P}_{x.a * x.b}" if hasattr(x, "P") else "")
def test_units_of_every_number_match_the_oracle(mc, oracle, spec, opts):
    m = mc.mc_model_create(spec, mc.mc_options_default(engine="config", **opts))
    assert mc.mc_count_states(m) == oracle.count(spec)
    t = oracle.min_time(spec)["t_min"]
    for prune, ee in ((1, 1), (0, 0), (0, 1), (1, 0)):
        mc.mc_set_options(m, mc.mc_options_default(engine="config", prune=prune, early_exit=ee, **opts))
        for T in (t - 1, t, 2 * t):
            exp = oracle.check(spec, T, prune=bool(prune), early_exit=bool(ee), widths=max(spec.n_workgroups) + 3)
            r = mc.mc_check(m, T)
            assert (r["holds"], r["states"], r["levels"]) == (exp["holds"], exp["states"], exp["levels"])
            assert mc.mc_last_widths(m) == exp["widths"]
            if not exp["holds"]:
                assert (r["cex_time"], r["cex_i"], r["cex_j"], r["cex_level"]) == (
                    exp["cex_time"], exp["cex_i"], exp["cex_j"], exp["cex_level"])
    for search in ("single", "lower"):
        mc.mc_set_options(m, mc.mc_options_default(engine="config", search=search, **opts))
        exp, r = oracle.min_time(spec, search=search), mc.mc_min_time(m)
        assert {k: r[k] for k in ("t_min", "t_ini", "states", "checks", "i", "j", "level")} == {
            k: exp[k] for k in ("t_min", "t_ini", "states", "checks", "i", "j", "level")}
