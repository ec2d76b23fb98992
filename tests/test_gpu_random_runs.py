"""Random runs on the GPU (T_ini and the swarm) against the oracle's
step-by-step runs: every number of units, both rules, runs of one work-group
and of hundreds, clocks of 32 and of 40 bits."""
import pytest

from paper_2305_09130_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def models():
    out = []
    for P in range(1, 17):
        for rule in (W.FREE, W.GREEDY):
            n_max = (1, 7, 40, 300)[(P + rule) % 4]
            m = W.random_small(8800 + 2 * P + rule, P, 3, 2, n_max, cost_max=9, speed_max=1 + P % 3, rule=rule,
                               key_bits=0 if P <= 4 else 128)
            most = 60 if rule == W.GREEDY else 9  # buffers of the exploration are sized with the model
            if P > 5:
                m.n_workgroups = [min(n, most) for n in m.n_workgroups]
            if P % 5 == 3:
                m.cost = [c + (1 << 31) // 7 for c in m.cost]
            out.append(m)
    return out


@pytest.mark.parametrize("spec", models(), ids=lambda s: f"{s.name}_P{s.P}_r{s.rule}")
def test_random_runs_match_oracle(mc, oracle, spec):
    m = mc.mc_model_create(spec)
    for seed, walks in ((1, 1), (2305091300, 5), (9, 1000)):
        assert mc.mc_simulate(m, seed, walks) == oracle.simulate(spec, seed, walks)
        got, exp = mc.mc_swarm(m, seed, walks, max_rounds=9, trace=False), oracle.swarm(spec, seed, walks, 9)
        for k in ("best_time", "first_time", "rounds", "walks", "best_walk", "i", "j"):
            assert got[k] == exp[k], (k, got, exp)
