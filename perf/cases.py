"""Performance cases of the explorer, through its public entry points.

Each case is one thing a user of the library has it do: a tuning query on a
small, a medium and a large model, exhaustive counts and certificate checks,
batches, served bursts, the swarm search, and the processing-element level
models.  A case holds plain sizes only; ``prepare`` draws the cost tables and
speeds from a seed and makes the handles a program keeps between queries, and
``run`` asks the query once.

Every output is a whole number (times, configurations, counts, packed
states), so outputs have to be equal; there are no rounded values.  A
counterexample's inner path is any valid one (several parents can reach a
state), so of a trace its length, its first states and its last are returned.
"""
from __future__ import annotations

import math

import numpy as np

from paper_2305_09130_gb300 import mc
from paper_2305_09130_gb300 import pe_workloads as PW
from paper_2305_09130_gb300 import workloads as W

MASK32 = (1 << 32) - 1


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: the tiny model's tuning query, trace included
        {"name": "c1_min_time", "kind": "min_time", "rule": "free", "P": 2, "G": 64, "a": 5, "b": 3,
         "cost": "table", "speed_max": 1, "key_bits": 0, "search": "single", "prune": 1, "trace": True},
        # an ordinary tuning query: G=1024 on four units of uneven speed
        {"name": "c2_min_time", "kind": "min_time", "rule": "greedy", "P": 4, "G": 1024, "a": 9, "b": 5,
         "cost": "formula", "speed_max": 3, "key_bits": 0, "search": "single", "prune": 1, "trace": False},
        # the large tuning query asked once: from host arrays to the answer
        {"name": "c3_query_from_arrays", "kind": "query", "rule": "greedy", "P": 8, "G": 4096, "a": 10, "b": 6,
         "cost": "table", "speed_max": 1, "key_bits": 128, "search": "single", "prune": 1, "trace": False},
        # exhaustive verification of the same model: every state counted
        {"name": "c3_count", "kind": "count", "rule": "greedy", "P": 8, "G": 4096, "a": 10, "b": 6,
         "cost": "table", "speed_max": 1, "key_bits": 128},
        # every interleaving on four units, 64-bit states, lowering without pruning
        {"name": "c2_star_lower", "kind": "min_time", "rule": "free", "P": 4, "G": 80, "a": 9, "b": 5,
         "cost": "formula", "speed_max": 3, "key_bits": 0, "search": "lower", "prune": 0, "trace": False},
        # odd sizes: certificate and counterexample checks at the optimum, with its trace
        {"name": "odd_free_certificate", "kind": "certify", "rule": "free", "P": 7, "G": 31, "a": 5, "b": 3,
         "cost": "table", "speed_max": 3, "key_bits": 0, "prune": 0},
        # the largest search: 1.07e9 states with 128-bit keys (the benchmark's headline)
        {"name": "c3_star_lower", "kind": "min_time", "rule": "free", "P": 8, "G": 36, "a": 10, "b": 6,
         "cost": "table", "speed_max": 1, "key_bits": 128, "search": "lower", "prune": 0, "trace": False},
        # many uneven models answered at once, checks and tuning queries mixed
        {"name": "c4_batch", "kind": "batch", "count": 256},
        # a burst of large tuning queries to the request loop
        {"name": "c5_served_burst", "kind": "served", "count": 48, "P": 8, "G": 4096, "a": 10, "b": 6},
        # the abstract kernel at the level of processing elements: wide levels
        {"name": "pe_abstract", "kind": "pe", "kernel": "abstract", "size": 16, "P": 4, "np": 4},
        # the Minimum kernel at that level: thousands of narrow levels
        {"name": "pe_minimum", "kind": "pe", "kernel": "minimum", "size": 64, "P": 4, "np": 4},
        # random runs for a first trail on the large model
        {"name": "c3_swarm", "kind": "swarm", "rule": "greedy", "P": 8, "G": 4096, "a": 10, "b": 6,
         "cost": "table", "speed_max": 1, "key_bits": 128, "walks": 262144},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_free(rng):
    """A FREE model of at most a drawn number of states (log-uniform)."""
    P = rng.randint(2, 8)
    a, b = rng.randint(3, 10), rng.randint(2, 6)
    target = math.exp(rng.uniform(math.log(1e3), math.log(2e8)))
    lo, hi = 2, 2048
    while lo < hi:  # the largest G with at most `target` states
        mid = (lo + hi + 1) // 2
        if _free_count({"P": P, "G": mid, "a": a, "b": b}) <= target:
            lo = mid
        else:
            hi = mid - 1
    return {"rule": "free", "P": P, "G": lo, "a": a, "b": b}


def _draw_greedy(rng):
    return {"rule": "greedy", "P": rng.randint(1, 10), "G": _log_uniform(rng, 33, 4096),
            "a": rng.randint(4, 10), "b": rng.randint(2, 6)}


def draw(rng):
    kind = rng.choice(["min_time", "min_time", "query", "count", "certify", "batch", "served", "pe", "swarm"])
    if kind == "batch":
        return {"kind": kind, "count": _log_uniform(rng, 8, 256)}
    if kind == "served":
        return {"kind": kind, "count": rng.randint(4, 48), "P": rng.randint(2, 8),
                "G": _log_uniform(rng, 257, 4096), "a": rng.randint(4, 10), "b": rng.randint(2, 6)}
    if kind == "pe":
        if rng.random() < 0.5:
            return {"kind": kind, "kernel": "abstract", "size": rng.choice([8, 16]), "P": rng.randint(1, 3),
                    "np": rng.randint(2, 4)}
        return {"kind": kind, "kernel": "minimum", "size": rng.choice([16, 32, 64]), "P": rng.randint(1, 4),
                "np": rng.randint(1, 4)}
    model = _draw_greedy(rng) if kind == "swarm" or rng.random() < 0.4 else _draw_free(rng)
    case = {"kind": kind, **model, "cost": "table", "cost_max": _log_uniform(rng, 256, 65536),
            "speed_max": rng.randint(1, 3), "key_bits": rng.choice([0, 128])}
    if kind in ("min_time", "query"):
        case.update(cost=rng.choice(["table", "formula"]), search=rng.choice(["single", "single", "lower", "bisect"]), prune=rng.choice([1, 1, 0]),
                    trace=rng.random() < 0.5)
        if case["search"] == "bisect":  # its holding checks would each explore everything
            case["prune"] = 1
    elif kind == "certify":
        case["prune"] = rng.choice([1, 0])
    elif kind == "swarm":
        case["walks"] = _log_uniform(rng, 1 << 10, 1 << 18)
    return case


# ---------------------------------------------------------------- inputs
def _spec(case, seed):
    """A model of the case's sizes with the seed's cost table and speeds."""
    rng = W.SplitMix64(seed * 1000003 + 17)
    P, G = case["P"], case["G"]
    wg, ts = W.pow2_range(0, case["a"] - 1), W.pow2_range(0, case["b"] - 1)
    speed = [rng.uniform(1, case.get("speed_max", 1)) for _ in range(P)]
    rule = W.FREE if case.get("rule") == "free" else W.GREEDY
    if case.get("cost") == "formula":
        spec = W.from_formula("perf", G, P, wg, ts, speed, rule)
    else:
        n = [W.n_workgroups_for(G, w) for w in wg for _ in ts]
        cost = [rng.uniform(1, case.get("cost_max", 16)) for _ in n]
        spec = W.ModelSpec("perf", P, wg, ts, n, cost, speed, rule, 0, G)
    if case["kind"] == "count":  # state counts follow the work-groups alone: with or without a ragged last one
        spec.n_workgroups = [max(1, n - rng.uniform(0, 1)) for n in spec.n_workgroups]
    spec.key_bits = case.get("key_bits", 0)
    return spec


def _optimum(spec):
    """The least terminal time of a model: the configuration's N-th completion
    when its work-groups are taken as early as possible (by bisection)."""
    best = None
    for n, cost in zip(spec.n_workgroups, spec.cost):
        lo, hi = 1, n * cost * min(spec.speed)
        while lo < hi:
            mid = (lo + hi) // 2
            if sum(mid // (cost * s) for s in spec.speed) >= n:
                hi = mid
            else:
                lo = mid + 1
        best = lo if best is None or lo < best else best
    return best


def _pe_spec(case, seed):
    """A processing-element level model; the seed draws each configuration's
    global-memory time."""
    rng = W.SplitMix64(seed * 1000003 + 29)
    size, P, np_ = case["size"], case["P"], case["np"]
    dom = [1 << e for e in range(1, size.bit_length() - 1)]
    n, pes, progs = [], [], []
    for w in dom:
        for t in dom:
            pes.append(min(w, np_))
            if case["kernel"] == "abstract":
                n.append(max(1, size // w))
                progs.append(PW.abstract_program(size, w, t, np_, rng.uniform(1, 2)))
            else:
                n.append(max(1, -(-size // (w * t))))
                progs.append(PW.minimum_program(w, t, np_, rng.uniform(1, 3)))
    return PW.PeSpec("perf_pe", P, dom, dom, n, pes, progs)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        specs = W.c4_instances(case["count"], seed=seed * 1000003 + 41)
        queries = []
        for s in specs:
            # thresholds around the optimum, as a tuner that has an estimate asks them
            rate = sum(1 / x for x in s.speed)
            near = min(n * c / rate for n, c in zip(s.n_workgroups, s.cost))
            queries.append(("min_time", None) if s.meta["query"] else
                           ("check", max(1, round(near * s.meta["t_frac_milli"] / 1000))))
        return {"kind": kind, "batch": mc.mc_batch_create(specs), "queries": queries}
    if kind == "served":
        specs = [_spec({**case, "key_bits": 128}, seed * 4099 + k) for k in range(case["count"])]
        return {"kind": kind, "server": mc.mc_server_create(slots=256, pool_bytes=4 << 30), "specs": specs}
    if kind == "pe":
        return {"kind": kind, "model": mc.mc_pe_model_create(_pe_spec(case, seed))}
    spec = _spec(case, seed)
    if kind == "query":
        return {"kind": kind, "spec": spec, "trace": case["trace"],
                "options": mc.mc_options_default(search=case["search"], prune=case["prune"], sim_seed=seed)}
    options = {k: case[k] for k in ("search", "prune") if k in case}
    if kind == "min_time":
        options["sim_seed"] = seed
    model = mc.mc_model_create(spec, mc.mc_options_default(**options))
    mc.mc_reserve(model)
    state = {"kind": kind, "model": model, "trace": case.get("trace", False)}
    if kind == "certify":
        state["T"] = _optimum(spec)
    elif kind == "swarm":
        state.update(seed=seed, walks=case["walks"])
    elif kind == "count":
        state["levels"] = case["G"] + 3
    return state


# ---------------------------------------------------------------- one pass
def _ints(*values):
    return np.array(values, dtype=np.int64)


def _key(k):
    """A packed state as 32-bit limbs."""
    return [(k >> s) & MASK32 for s in (0, 32, 64, 96)]


def _trace_ends(trace):
    ends = [0] * 4 if not trace else trace[:3] + trace[-1:]
    return _ints(len(trace or []), *(x for k in ends for x in _key(k)))


def _min_time(r, trace):
    out = {"answer": _ints(r["t_min"], r["t_ini"], r["wg"], r["ts"], r["states"], r["checks"], r["level"]),
           "witness": _ints(*_key(r["witness_key"]))}
    if trace:
        out["trace"] = _trace_ends(r["trace"])
    return out


def _check(r):
    return {"answer": _ints(r["holds"], r["states"], r["levels"], r.get("cex_time", 0), r.get("cex_wg", 0),
                            r.get("cex_ts", 0), r.get("cex_level", 0), *_key(r.get("cex_key", 0))),
            "trace": _trace_ends(r.get("trace"))}


_ANSWER = ("status", "holds", "levels", "states", "checks", "level", "time", "t_ini", "wg", "ts")


def _answers(results):
    out = {f: _ints(*(int(r[f]) for r in results)) for f in _ANSWER}
    out["key"] = np.array([_key(r["key"]) for r in results], dtype=np.int64)
    return out


def run(state):
    kind = state["kind"]
    if kind == "min_time":
        return _min_time(mc.mc_min_time(state["model"], trace=state["trace"]), state["trace"])
    if kind == "query":
        model = mc.mc_model_create(state["spec"], state["options"], allocator="cuda")
        out = _min_time(mc.mc_min_time(model, trace=state["trace"]), state["trace"])
        mc.mc_model_destroy(model)
        return out
    if kind == "count":
        states = mc.mc_count_states(state["model"])
        widths = np.zeros(state["levels"], dtype=np.int64)
        got = mc.mc_last_widths(state["model"], state["levels"])
        widths[:len(got)] = got
        return {"states": states, "widths": widths}
    if kind == "certify":
        return [_check(mc.mc_check(state["model"], state["T"] - 1)), _check(mc.mc_check(state["model"], state["T"]))]
    if kind == "batch":
        return _answers(mc.mc_batch_run(state["batch"], state["queries"]))
    if kind == "served":
        server, got = state["server"], []
        for spec in state["specs"]:
            mc.mc_server_submit(server, spec, "min_time")
        while len(got) < len(state["specs"]):
            got += mc.mc_server_poll(server, wait_ms=100)
        return _answers(sorted(got, key=lambda r: r["ticket"]))
    if kind == "pe":
        r = mc.mc_pe_min_time(state["model"], trace=False)
        return {"answer": _ints(r["t_min"], r["wg"], r["ts"], r["states"], r["checks"], r["level"]),
                "witness": _ints(*_key(r["witness_key"]))}
    r = mc.mc_swarm(state["model"], state["seed"], state["walks"], max_rounds=16, trace=False)
    return _ints(r["best_time"], r["first_time"], r["wg"], r["ts"], r["rounds"], r["walks"], r["best_walk"])


# ---------------------------------------------------------------- least work
def _free_count(case):
    """Reachable states under FREE: C(N + P, P) per configuration."""
    return 1 + case["a"] + case["b"] * sum(math.comb(W.n_workgroups_for(case["G"], 1 << i) + case["P"], case["P"])
                                           for i in range(case["a"]))


def _greedy_states(spec, T=None):
    """Reachable states under GREEDY (of time at most T): while one instant's
    starts are handed out, every subset of the units that start then."""
    total = 1 + spec.a + spec.a * spec.b
    for n, cost in zip(spec.n_workgroups, spec.cost):
        t = [cost * s for s in spec.speed]
        clk, left = [0] * spec.P, n
        while left:
            now = min(clk)
            tied = [c for c in range(spec.P) if clk[c] == now]
            fit = [c for c in tied if T is None or now + t[c] <= T]
            total += sum(math.comb(len(fit), x) for x in range(1, min(left, len(fit)) + 1))
            if len(fit) < len(tied) or left <= len(tied):
                break
            left -= len(tied)
            for c in tied:
                clk[c] += t[c]
    return total


def _states(case):
    """Unique states the query cannot do without: every reachable one for an
    exhaustive search, those of time at most the optimum where pruning may
    drop the rest."""
    if case["rule"] == "free":
        if not case.get("prune"):
            return _free_count(case)
        spec = _spec(case, 1)
        T = _optimum(spec)
        # the box of work-groups each unit finishes by the optimum, below N
        return 1 + case["a"] + sum(min(math.comb(n + spec.P, spec.P), math.prod(T // (c * s) + 1 for s in spec.speed))
                                   for n, c in zip(spec.n_workgroups, spec.cost))
    spec = _spec(case, 1)
    return _greedy_states(spec, _optimum(spec) if case.get("prune") else None)


def work(case):
    """Bytes: each unique state's key written once, and the tables read and
    answers written.  Operations: one clock update and one comparison per unit
    for each unique state (or each dispatch of a random run)."""
    kind = case["kind"]
    if kind == "batch":
        specs = W.c4_instances(case["count"], seed=1000003 + 41)
        states = sum(_greedy_states(s, _optimum(s)) for s in specs)
        return {"bytes": 16 * states + 400 * case["count"], "flops": 2 * 8 * states}
    if kind == "served":
        states = sum(_states({**case, "rule": "greedy", "prune": 1}) for _ in range(case["count"]))
        return {"bytes": 16 * states + 400 * case["count"], "flops": 2 * case["P"] * states}
    if kind == "pe":
        spec = _pe_spec(case, 1)
        # a unit's program alone: its steps' subsets of marked PEs, per work-group
        states = sum(n * sum((2 ** m) * max(1, t) for t, m in prog) for n, prog in zip(spec.n_workgroups, spec.programs))
        return {"bytes": 16 * states * case["P"], "flops": 2 * case["P"] * case["np"] * states}
    if kind == "swarm":
        n = sum(W.n_workgroups_for(case["G"], 1 << i) for i in range(case["a"])) / case["a"]
        steps = int(case["walks"] * n)
        return {"bytes": 8 * case["a"] * case["b"] + 64, "flops": 2 * case["P"] * steps}
    states = _states(case)
    return {"bytes": (16 if case["key_bits"] == 128 else 8) * states, "flops": 2 * case["P"] * states}


def exact(case, seed):
    """Every output is a whole number and has to be equal: no value is rounded."""
    return None
