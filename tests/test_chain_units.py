"""Chain units: FREE configurations of two to four units explored chain by
chain (the states that share the counts of all units but the last), and their
trace, rebuilt from the witness's counts.

On the CPU the chains are restated and compared with the oracle's general
search; on the GPU the configuration engine is compared with the oracle and
with the level engine."""
import itertools

import pytest

import closed_forms as CF
import replay as RP
from paper_2305_09130_gb300 import workloads as W

NO_LIMIT = (1 << 64) - 1


def chains(P, N, t, T, prune):
    """Widths of a configuration's levels below its select state, and its
    least violating terminal (time, counts)."""
    most = [min(N, T // x) if prune else N for x in t]
    widths, worst = [0] * (N + 1), None
    for head in itertools.product(*(range(m + 1) for m in most[:-1])):
        taken = sum(head)
        for k in range(taken, min(N, taken + most[-1]) + 1):
            widths[k] += 1
            if k == N:
                counts = head + (N - taken,)
                time = max(n * x for n, x in zip(counts, t))
                if time <= T and (worst is None or (time, counts) < worst):
                    worst = (time, counts)
    return widths[1:], worst


def models():
    out = []
    for P in (2, 3, 4):
        for speed_max in (1, 3):
            out.append(W.random_small(8100 + 10 * P + speed_max, P, 2, 2, 14 - 2 * P, cost_max=5, speed_max=speed_max))
    return out


@pytest.mark.parametrize("spec", models(), ids=lambda s: f"{s.name}_P{s.P}")
def test_chains_are_the_general_search(oracle, spec):
    t_min = oracle.min_time(spec)["t_min"]
    for T in sorted({0, t_min - 1, t_min, t_min + 2, NO_LIMIT}):
        for prune in (False, True):
            exp = oracle.check(spec, T, prune=prune, early_exit=False)
            states, worst = 1 + spec.a + spec.a * spec.b, None
            for k, (N, cost) in enumerate(zip(spec.n_workgroups, spec.cost)):
                widths, w = chains(spec.P, N, [cost * s for s in spec.speed], T, prune)
                states += sum(widths)
                if w is not None:
                    cand = (2 + N, w[0], k // spec.b, k % spec.b, w[1])
                    worst = cand if worst is None or cand < worst else worst
            assert states == exp["states"]
            assert (worst is None) == exp["holds"]
            if worst:
                assert worst == (exp["cex_level"], exp["cex_time"], exp["cex_i"], exp["cex_j"], tuple(exp["cex_n"]))


def gpu_models():
    """Two to four units, and one and five (their neighbours on the other
    units); shallow and deep configurations side by side, a depth at which a
    level outgrows a warp and the widest a block takes, both key widths, clocks
    of 32 and of 40 bits."""
    out = []
    for P, N in ((1, 40), (2, 64), (2, 255), (3, 17), (3, 40), (4, 6), (4, 16), (5, 6)):
        spec = W.random_small(8200 + 10 * P + N, P, 2, 2, N, cost_max=6, speed_max=3, key_bits=128 if N % 2 else 0)
        spec.n_workgroups = [N, N - 1, 1, N // 2]
        out.append(spec)
    big = W.random_small(8290, 3, 2, 2, 12, cost_max=5, speed_max=2)
    big.cost = [c + (1 << 31) for c in big.cost]  # clocks beyond 32 bits
    out.append(big)
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("spec", gpu_models(), ids=lambda s: f"{s.name}_P{s.P}_k{s.key_bits}_N{max(s.n_workgroups)}")
def test_chain_units_match_oracle_and_levels(mc, oracle, spec):
    t_min = oracle.min_time(spec)["t_min"]
    opts = [{}, {"unit_threads": 64}, {"unit_threads": 512}]
    models = [mc.mc_model_create(spec, mc.mc_options_default(engine="config", **o)) for o in opts]
    level = mc.mc_model_create(spec, mc.mc_options_default(engine="level"))
    lay = mc.mc_model_layout(models[0])
    for m in models:
        assert mc.mc_count_states(m) == CF.count(spec)
        assert mc.mc_last_widths(m) == CF.widths(spec)
    for T in (0, t_min - 1, t_min, t_min + 1, 2 * t_min, NO_LIMIT):
        for prune, ee in ((1, 1), (0, 1), (1, 0), (0, 0)):
            exp = oracle.check(spec, T, prune=bool(prune), early_exit=bool(ee))
            mc.mc_set_options(level, mc.mc_options_default(engine="level", prune=prune, early_exit=ee))
            trace = mc.mc_check(level, T).get("trace")
            for m, o in zip(models, opts):
                mc.mc_set_options(m, mc.mc_options_default(engine="config", prune=prune, early_exit=ee, **o))
                r = mc.mc_check(m, T)
                assert (r["holds"], r["states"], r["levels"]) == (exp["holds"], exp["states"], exp["levels"])
                assert mc.mc_last_widths(m) == mc.mc_last_widths(level)
                if not exp["holds"]:
                    i, j, n = RP.decode(lay, r["cex_key"])
                    assert (r["cex_time"], i - 1, j - 1, r["cex_level"], n) == (
                        exp["cex_time"], exp["cex_i"], exp["cex_j"], exp["cex_level"], exp["cex_n"])
                    assert r["trace"] == trace
                    RP.replay(spec, lay, r["trace"], lambda t: t <= T)
    for search in ("single", "lower", "bisect"):
        exp = oracle.min_time(spec, search=search, prune=True)
        mc.mc_set_options(models[0], mc.mc_options_default(engine="config", search=search))
        r = mc.mc_min_time(models[0])
        assert {k: r[k] for k in ("t_min", "t_ini", "states", "checks", "i", "j", "level")} == \
            {k: exp[k] for k in ("t_min", "t_ini", "states", "checks", "i", "j", "level")}
        RP.replay(spec, lay, r["trace"], lambda t: t == r["t_min"])
