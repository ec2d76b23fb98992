"""mc_layout says what the passes use, memory is set aside for what they use,
and the tuner's candidates differ in what they read (no device needed)."""
import pytest

import bench
from paper_2305_09130_gb300 import autotune as AT
from paper_2305_09130_gb300 import mc
from paper_2305_09130_gb300 import workloads as W


@pytest.fixture(scope="module")
def lib():
    return mc.load()


def layout(spec, **kw):
    return mc.mc_model_layout(mc.mc_model_create(spec, mc.mc_options_default(engine="level", **kw), allocator=None))


@pytest.mark.parametrize("n,used,general,ordered", [(7, 26, 16, 16), (63, 50, 16, 14), (127, 58, 16, 16)])
def test_log_tag_bits_of_narrow_128_bit_keys(lib, n, used, general, ordered):
    """Ordered expansion keeps 128-bit keys of at most 56 used bits in the low
    word, tag above it: 64 - used bits at most.  A pass that probes a visited
    set, and keys of more used bits, spread the key over both words."""
    spec = W.ModelSpec("narrow", 8, [1], [1], [n], [1], [1] * 8, key_bits=128)
    assert layout(spec)["used_bits"] == used
    assert layout(spec)["log_tag_bits"] == ordered
    assert layout(spec, probe_scheme="split")["log_tag_bits"] == general
    assert layout(spec.with_rule(W.GREEDY))["log_tag_bits"] == general
    assert layout(spec, no_log_tags=1)["log_tag_bits"] == 0


def test_log_tag_bits_of_c3_star(lib):
    lay = layout(W.c3_star())
    assert (lay["used_bits"], lay["log_tag_bits"]) == (55, 9)


def test_pe_candidates_differ_in_what_the_ordered_pass_reads():
    assert set(AT.PE_SPACE) == {"blocks_per_sm"}
    cands = AT.candidates(AT.PE_SPACE)
    assert len({c["blocks_per_sm"] for c in cands}) == len(cands) == 3


@pytest.mark.parametrize("spec,opts,keeps", [(W.c3(), {}, False), (W.c3(), {"unit_threads": 128}, True),
                                             (W.c2(), {}, False), (W.c1(W.FREE), {}, False),
                                             (W.c1(W.FREE), {"unit_threads": 64}, False),
                                             (W.random_small(91, 11, 2, 2, 30, rule=W.GREEDY), {}, True)],
                         ids=lambda x: getattr(x, "name", None) or str(x))
def test_log_memory_only_where_units_keep_a_log(lib, spec, opts, keeps):
    """Configuration engine: block units of GREEDY models keep a frontier log;
    warps and FREE units do not, and nothing is set aside for one."""
    o = mc.mc_options_default(engine="config", **opts)
    spec = spec.with_key_bits(128)
    lay = mc.mc_model_layout(mc.mc_model_create(spec, o, allocator=None))
    log = 20 * lay["log_capacity"]
    assert log > 0 and (lay["device_bytes"] > log) == keeps
    batch = mc.mc_batch_create([spec], o, allocator=None)
    size = mc.mc_batch_device_bytes(batch)
    mc.mc_batch_destroy(batch)
    assert (size > log) == keeps
    assert bench.config_units(spec, lay, o)[1] == keeps


def test_bench_names_what_explores_a_configuration(lib):
    def units(spec, **kw):
        o = mc.mc_options_default(engine="config", **kw)
        return bench.config_units(spec, mc.mc_model_layout(mc.mc_model_create(spec, o, allocator=None)), o)[0]

    assert "wave units" in units(W.c3()) and "wave units" in units(W.c2()) and "u128" in units(W.c3())
    assert units(W.c3(), unit_threads=128) == "cfg_kernel<u128> (128 threads per configuration)"
    assert units(W.c1(W.FREE)) == "cfg_kernel<u64> (chain units, 256 threads per configuration)"
    assert units(W.random_small(92, 1, 2, 2, 9)) == "cfg_warp_kernel<u64> (a warp per configuration)"
    assert "threads per configuration" in units(W.random_small(91, 11, 2, 2, 30, rule=W.GREEDY))
