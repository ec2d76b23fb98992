"""Random runs in numbers from which each takes a lane instead of a warp: T_ini
equals the oracle's just below and just above those numbers, in queries and in
batches."""
import pytest

from paper_2305_09130_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def models():
    out = [W.random_small(9100 + P, P, 3, 2, (40, 5, 300)[P % 3] if P < 5 else 6, rule=rule, speed_max=4)
           for P, rule in ((1, W.GREEDY), (2, W.FREE), (3, W.GREEDY), (4, W.GREEDY), (6, W.FREE), (8, W.GREEDY),
                           (10, W.GREEDY), (16, W.GREEDY))]
    big = W.random_small(9150, 5, 2, 2, 8, rule=W.GREEDY)
    big.cost = [c + (1 << 30) for c in big.cost]
    return out + [big]


@pytest.mark.parametrize("spec", models(), ids=lambda s: f"{s.name}_P{s.P}_r{s.rule}")
def test_many_runs_match_the_oracle(mc, oracle, spec):
    m = mc.mc_model_create(spec)
    for walks in (8191, 8192, 8200) if spec.rule == W.GREEDY else (8192, 131071, 131072, 131100):
        for seed in (3, 2305091300):
            assert mc.mc_simulate(m, seed, walks) == oracle.simulate(spec, seed, walks)


@pytest.mark.parametrize("walks", [1, 33, 1023, 1024, 16383, 16384])  # (times eight models: the numbers above)
def test_many_runs_in_a_batch(mc, oracle, walks):
    specs = [s for s in models() if s.P < 16]  # (a level of the 16 units does not fit a block)
    assert len(specs) == 8
    b = mc.mc_batch_create(specs, mc.mc_options_default(sim_walks=walks, engine="config"))
    results = mc.mc_batch_run(b, [("min_time", None)] * len(specs))
    st = mc.mc_batch_get_stats(b)
    mc.mc_batch_destroy(b)
    for r, spec in zip(results, specs):
        e = oracle.min_time(spec, walks=walks)
        assert (r["status"], r["t_ini"], r["time"], r["states"]) == (0, e["t_ini"], e["t_min"], e["states"])
    # clear, simulate, two passes, and the launch for runs that take a lane each
    assert st["explore_launches"] + st["other_launches"] == 4 + (walks * len(specs) >= 8192)
