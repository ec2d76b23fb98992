"""Ordered expansion of the PE-level model: since the last tick, a unit acts
only when no later unit has acted, and marks by PE index, so every state is
generated once and no visited set is kept.

The rule is restated on the brute force's states and compared with its full
search, level by level; on the GPU the ordered pass is compared with the pass
that keeps a visited set, and with the oracle."""
import pytest

import pe_bruteforce as PB
from paper_2305_09130_gb300 import pe_workloads as PW
from test_pe_oracle_pins import random_pe, tiny_pe_models

NO_LIMIT = (1 << 64) - 1


def ordered_successors(M, s):
    if len(s) != 7:
        return M.successors(s)
    i, j, n, busy, pc, mask, t = s
    cfg = i * M.spec.b + j
    steps = M.steps[cfg]
    ticks = [sum(k == "W" for k, _m in steps[:x]) for x in range(len(steps) + 1)]
    acted = -1
    for c in range(M.P):
        if busy[c]:
            entered = pc[c] == 0 or steps[pc[c] - 1][0] == "B"
            if mask[c] or entered:
                acted = c
        elif n[c] and steps[-1][0] == "B" and n[c] * ticks[-1] == t:
            acted = c
    out = []
    for x in M.successors(s):
        changed = [c for c in range(M.P) if (n[c], busy[c], pc[c], mask[c]) != (x[2][c], x[3][c], x[4][c], x[5][c])]
        if x[6] == t:  # an event of one unit
            (c,) = changed
            new = x[5][c] & ~mask[c]
            if c < acted or (new and new < mask[c]):
                continue
        out.append(x)
    return out


def more_models():
    """Programs that end at a barrier, barriers in a row, one PE, a unit more
    than there are work-groups."""
    prog = [[(1, 2), (0, 2)], [(0, 1), (0, 2), (1, 1), (0, 2)], [(2, 1), (0, 1)], [(1, 2), (0, 1), (1, 1)]]
    return [PW.PeSpec("ends_at_barriers", 2, [1, 2], [1, 2], [3, 2, 1, 4], [2, 2, 1, 2], prog),
            PW.PeSpec("three_units", 3, [1], [1, 2], [2, 4], [2, 1], [prog[0], prog[2]]),
            PW.PeSpec("no_ticks", 2, [1], [1], [3], [2], [[(0, 2), (0, 1)]])]


@pytest.mark.parametrize("spec", tiny_pe_models() + more_models(), ids=lambda s: f"{s.name}_P{s.P}")
def test_ordered_generation_is_the_full_search(spec):
    M = PB.PeModel(spec)
    full = PB.enumerate_levels(spec)
    times = sorted({M.time(s) for lv in full for s in lv})
    for T in {times[-1], times[len(times) // 2], 0}:
        level, got = [("s0",)], []
        while level:
            got.append(level)
            level = [x for s in level for x in ordered_successors(M, s) if M.time(x) <= T]
            assert len(level) == len(set(level))
        exp, cur = [], {("s0",)}
        while cur:
            exp.append(cur)
            cur = {x for s in cur for x in M.successors(s) if M.time(x) <= T}
        assert [set(x) for x in got] == exp


def gpu_models():
    """Unit fields that fit the key's low word and that do not; levels handled
    by one block, by all, and back."""
    out = more_models()[:2] + [PW.pe_abstract(8, P=3, np_=2), PW.pe_minimum(32, P=4, np_=4, gmt=2), PW.pe_minimum(16, P=1, np_=1, gmt=1),
                           random_pe(7511, 5, 2, 1, n_max=2, nwe_max=2), random_pe(7512, 2, 1, 2, n_max=5, nwe_max=4)]
    wide = PW.pe_abstract(8, P=4, np_=2)  # 17-bit unit fields at P = 4: 68 bits
    wide.n_workgroups = [n if k else 40 for k, n in enumerate(wide.n_workgroups)]
    return out + [wide]


@pytest.mark.gpu
@pytest.mark.parametrize("spec", gpu_models(), ids=lambda s: f"{s.name}_P{s.P}")
def test_ordered_pass_matches_visited_set(mc, spec):
    opts = [{"max_probes": 64}, {}, {"no_log_tags": 1}, {"threads_per_block": 64, "blocks_per_sm": 1}]
    models = [mc.mc_pe_model_create(spec, mc.mc_options_default(**o)) for o in opts]
    counts = [mc.mc_pe_count_states(m) for m in models]
    widths = [mc.mc_pe_last_widths(m) for m in models]
    assert counts == [counts[0]] * len(opts) and widths == [widths[0]] * len(opts)
    t_min = mc.mc_pe_min_time(models[0], trace=False)["t_min"]
    for prune, ee in ((1, 1), (0, 1), (1, 0), (0, 0)):
        ms = [mc.mc_pe_model_create(spec, mc.mc_options_default(prune=prune, early_exit=ee, **o)) for o in opts]
        for T in (0, t_min - 1, t_min, t_min + 3, NO_LIMIT):
            rs = [mc.mc_pe_check(m, T) for m in ms]
            ws = [mc.mc_pe_last_widths(m) for m in ms]
            lay = mc.mc_pe_model_layout(ms[0])
            for r, w in zip(rs, ws):
                assert {k: v for k, v in r.items() if k != "trace"} == {k: v for k, v in rs[0].items() if k != "trace"}
                assert w == ws[0]
                if not r["holds"]:
                    from test_gpu_pe import replay
                    replay(spec, lay, r["trace"], T)
        answers = [mc.mc_pe_min_time(m) for m in ms]
        for r in answers:
            assert {k: v for k, v in r.items() if k != "trace"} == {k: v for k, v in answers[0].items() if k != "trace"}
