"""Requests of a server with pruning off: GREEDY models whose levels fit a warp
(wave units), wider ones (block units) and FREE ones, against the oracle."""
import pytest

import replay as RP
from paper_2305_09130_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def specs():
    out = [W.c1(W.GREEDY), W.c2(rule=W.GREEDY), W.c1(W.FREE)]
    return out + [W.random_small(8800 + P, P, 2, 3, 90, speed_max=2, rule=W.GREEDY) for P in (1, 4, 5, 8, 10, 11)]


def test_requests_without_pruning_match_the_oracle(mc, oracle):
    srv = mc.mc_server_create(slots=16, pool_bytes=2 << 30, options=mc.mc_options_default(prune=0))
    asked = {}
    for spec in specs():
        exp = oracle.min_time(spec, prune=False)
        asked[mc.mc_server_submit(srv, spec, "min_time")] = (spec, None, exp)
        for T in (exp["t_min"] - 1, exp["t_min"] + 5):
            asked[mc.mc_server_submit(srv, spec, "check", T)] = (spec, T, oracle.check(spec, T, prune=False))
    got = {}
    while len(got) < len(asked):
        got.update({r["ticket"]: r for r in mc.mc_server_poll(srv, wait_ms=1000)})
    for ticket, (spec, T, exp) in asked.items():
        r = got[ticket]
        n = RP.decode(mc.mc_model_layout(mc.mc_model_create(spec.with_key_bits(128))), r["key"])[2]
        assert r["status"] == 0 and r["path"] == "config" and r["states"] == exp["states"]
        if T is None:
            assert {k: r[k] for k in ("t_ini", "checks", "i", "j", "level")} == {
                k: exp[k] for k in ("t_ini", "checks", "i", "j", "level")}
            assert (r["time"], list(n)) == (exp["t_min"], exp["n"])
        elif exp["holds"]:
            assert r["holds"] and r["levels"] == exp["levels"]
        else:
            assert (r["time"], r["i"], r["j"], r["level"], list(n)) == (
                exp["cex_time"], exp["cex_i"], exp["cex_j"], exp["cex_level"], exp["cex_n"])
    mc.mc_server_destroy(srv)
