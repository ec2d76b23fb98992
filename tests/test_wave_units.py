"""Wave units: GREEDY configurations explored with a level as a bitmap over
the subsets of the units that start together.

On the CPU the bitmap algorithm is restated step by step and compared with
the oracle's general search; on the GPU the wave units are compared with the
oracle and with the block units over every number of units they take, and one
more (which takes blocks)."""
import random

import pytest

import closed_forms as CF
import replay as RP
from paper_2305_09130_gb300 import workloads as W

NO_LIMIT = (1 << 64) - 1


def wave_unit(P, N, t, T, prune):
    """One configuration: (widths of levels 3.., least violating time, its
    smallest counts).  Positions: the units of E in descending index."""
    clk, n, total, widths = [0] * P, [0] * P, 0, []
    while True:
        mn = min(clk)
        E = [c for c in range(P - 1, -1, -1) if clk[c] == mn]
        A = sum(1 << q for q, c in enumerate(E) if not (prune and clk[c] + t[c] > T))
        m = min(N - total, bin(A).count("1"))
        cur = 1  # bit s: subset s is in the level
        for _ in range(m):
            nxt = 0
            for q in range(len(E)):
                if (A >> q) & 1:
                    lacks = sum(1 << s for s in range(1 << len(E)) if not (s >> q) & 1)
                    nxt |= (cur & lacks) << (1 << q)
            cur = nxt
            widths.append(bin(cur).count("1"))
        total += m
        if total == N or m < len(E):
            break
        for c in E:
            clk[c] += t[c]
            n[c] += 1
    if total < N:
        return widths, None, None
    best = None
    for s in range(1 << len(E)):
        if (cur >> s) & 1:
            time = max(clk + [clk[c] + t[c] for q, c in enumerate(E) if (s >> q) & 1])
            if time <= T and (best is None or time < best[0]):
                best = (time, tuple(n[c] + (c in E and (s >> E.index(c)) & 1) for c in range(P)))
    return (widths,) + (best or (None, None))


def models():
    rng = random.Random(5)
    out = []
    for P in (1, 2, 3, 5, 6, 8):
        for smax in (1, 3):
            out.append(W.random_small(7100 + 10 * P + smax, P, 2, 2, rng.randint(3, 17), cost_max=6, speed_max=smax,
                                      rule=W.GREEDY))
    return out


@pytest.mark.parametrize("spec", models(), ids=lambda s: f"{s.name}_P{s.P}")
def test_bitmap_levels_match_the_general_search(oracle, spec):
    t_min = oracle.min_time(spec)["t_min"]
    for T in sorted({0, t_min - 1, t_min, t_min + 2, 2 * t_min, NO_LIMIT}):
        for prune in (False, True):
            exp = oracle.check(spec, T, prune=prune, early_exit=False)
            states, worst = 1 + spec.a + spec.a * spec.b, None
            for k, (N, cost) in enumerate(zip(spec.n_workgroups, spec.cost)):
                w, time, counts = wave_unit(spec.P, N, [cost * s for s in spec.speed], T, prune)
                states += sum(w)
                if time is not None:
                    cand = (2 + N, time, k // spec.b, k % spec.b, counts)
                    worst = cand if worst is None or cand < worst else worst
            assert states == exp["states"]
            assert (worst is None) == exp["holds"]
            if worst:
                assert worst == (exp["cex_level"], exp["cex_time"], exp["cex_i"], exp["cex_j"], tuple(exp["cex_n"]))


def gpu_models():
    """Every P the wave units take (1..10: one to 32 words of subsets) and 11;
    equal speeds (all units start together) and uneven ones, both key widths,
    clocks of 32 and of 40 bits."""
    out = []
    for P in range(1, 12):
        out.append(W.random_small(7300 + P, P, 2, 3, 13 if P < 9 else 11, cost_max=5, speed_max=1, rule=W.GREEDY,
                                  key_bits=128 if P % 2 else 0))
        out.append(W.random_small(7330 + P, P, 2, 2, 19 if P < 9 else 12, cost_max=7, speed_max=3, rule=W.GREEDY))
    # hundreds of levels, waves of one unit and of several mixed (the widths of
    # one-state levels are added 32 levels at a time)
    # (and several segments of a configuration, their borders inside waves)
    for P, speed in ((2, [2, 3]), (3, [2, 3, 3]), (5, [1, 2, 2, 3, 3]), (6, [2] * 6)):
        deep = W.random_small(7390 + P, P, 2, 2, 300, cost_max=5, rule=W.GREEDY)
        deep.speed = speed
        deep.n_workgroups = [300, 257, 33, 100]
        out.append(deep)
    wide = W.random_small(7399, 6, 2, 2, 17, cost_max=5, speed_max=2, rule=W.GREEDY)
    wide.cost = [c + (1 << 32) // 3 for c in wide.cost]  # clocks beyond 32 bits
    out.append(wide)
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("spec", gpu_models(), ids=lambda s: f"{s.name}_P{s.P}_k{s.key_bits}")
def test_wave_units_match_oracle_and_blocks(mc, oracle, spec):
    t_min = oracle.min_time(spec)["t_min"]
    wave = mc.mc_model_create(spec, mc.mc_options_default(engine="config"))
    block = mc.mc_model_create(spec, mc.mc_options_default(engine="config", unit_threads=64))
    lay = mc.mc_model_layout(wave)
    for m in (wave, block):
        assert mc.mc_count_states(m) == oracle.count(spec)
        assert mc.mc_last_widths(m) == CF.widths(spec)
    for T in (0, t_min - 1, t_min, t_min + 1, 2 * t_min, NO_LIMIT):
        for prune, ee in ((1, 1), (0, 1), (1, 0), (0, 0)):
            exp = oracle.check(spec, T, prune=bool(prune), early_exit=bool(ee))
            got = []
            for m in (wave, block):
                mc.mc_set_options(m, mc.mc_options_default(prune=prune, early_exit=ee))
                got.append(mc.mc_check(m, T))
            assert mc.mc_last_widths(wave) == mc.mc_last_widths(block)
            for r in got:
                assert (r["holds"], r["states"], r["levels"]) == (exp["holds"], exp["states"], exp["levels"])
                if not exp["holds"]:
                    i, j, n = RP.decode(lay, r["cex_key"])
                    assert (r["cex_time"], i - 1, j - 1, r["cex_level"], n) == (
                        exp["cex_time"], exp["cex_i"], exp["cex_j"], exp["cex_level"], exp["cex_n"])
                    assert r["trace"][-1] == r["cex_key"] and len(r["trace"]) == r["cex_level"] + 1
                    RP.replay(spec, lay, r["trace"], lambda t: t <= T)
    for search in ("single", "lower", "bisect"):
        for prune in (1, 0):
            exp = oracle.min_time(spec, search=search, prune=bool(prune))
            mc.mc_set_options(wave, mc.mc_options_default(prune=prune, search=search))
            r = mc.mc_min_time(wave)
            assert {k: r[k] for k in ("t_min", "t_ini", "states", "checks", "i", "j", "level")} == \
                {k: exp[k] for k in ("t_min", "t_ini", "states", "checks", "i", "j", "level")}
            assert RP.decode(lay, r["witness_key"])[2] == exp["n"]
            RP.replay(spec, lay, r["trace"], lambda t: t == r["t_min"])


def run_models():
    """Models of a run: configurations of one and of several segments (512
    work-groups), waves on their borders; a FREE model and an 11-unit one
    beside them."""
    out = []
    for P, speed, N in ((6, [2] * 6, [1537, 512, 513, 5]), (5, [1, 2, 2, 3, 3], [1300, 1024, 40, 511]),
                        (2, [2, 3], [2048, 700, 512, 1])):
        deep = W.random_small(7420 + P, P, 2, 2, max(N), cost_max=5, rule=W.GREEDY, key_bits=128)
        deep.speed, deep.n_workgroups = speed, N
        out.append(deep)
    out.append(W.random_small(7430, 3, 2, 2, 9, cost_max=5, speed_max=2, key_bits=128))
    out.append(W.random_small(7431, 11, 2, 2, 9, cost_max=5, speed_max=2, rule=W.GREEDY, key_bits=128))
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("prune", (1, 0))
def test_runs_in_segments_match_single_models(mc, prune):
    specs = run_models()
    opt = mc.mc_options_default(engine="config", prune=prune, search="single")
    models = [mc.mc_model_create(s, opt) for s in specs]
    mins = [mc.mc_min_time(m) for m in models]
    batch = mc.mc_batch_create(specs, mc.mc_options_default(prune=prune))
    for shift in (None, -1, 0, 1):
        queries = [("min_time", None) if shift is None else ("check", m["t_min"] + shift) for m in mins]
        for k, (r, m, q) in enumerate(zip(mc.mc_batch_run(batch, queries), models, queries)):
            exp = mins[k] if shift is None else mc.mc_check(m, q[1])
            assert (r["status"], r["states"]) == (0, exp["states"])
            if shift is None or not exp["holds"]:
                time, key = ("t_min", "witness_key") if shift is None else ("cex_time", "cex_key")
                assert (r["time"], r["key"]) == (exp[time], exp[key])
                assert mc.mc_batch_trace(batch, k) == exp["trace"]
    mc.mc_batch_destroy(batch)
