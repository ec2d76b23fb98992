"""Orders that the device code keeps and that no run can show broken without
harm: read from the sources, with the arithmetic that makes them necessary
restated here."""
import os
import re

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2305_09130_gb300", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def between(text, start, end):
    at = text.index(start)
    return text[at:text.index(end, at)]


def test_narrow_levels_decode_only_entries_that_appeared():
    """A log entry that does not appear within the wait limit leaves a raw word
    behind.  Decoded, an untouched (zero) word names configuration -1 of -1:
    an index far outside the configuration table.  So the pass over narrow
    levels ends before it decodes anything when an entry failed, as the pass
    over wide levels skips such an entry."""
    a, b = 10, 6
    i = j = (0 - 1) & 0xFFFFFFFF
    assert (i * b + j) & 0xFFFFFFFF >= a * b
    text = source("mc_pe_ordered.cuh")
    narrow = between(text, "if (blockIdx.x == 0)", "while (!end)")
    load, after = narrow.split("__syncthreads();", 1)
    assert re.search(r"if \(!entry\(.*s_flags = kPeFlagError;", load)
    assert re.search(r"if \(s_flags & kPeFlagError\) end = 1;", after)
    for call in re.finditer(r"pe_slots<PT, SMALL>\(p, own", text):  # wide levels: behind the check
        assert "if (entry(" in text[:call.start()].rsplit("if (s < Wl)", 1)[1]


def test_a_warps_widths_are_ordered_before_its_completion():
    """Lanes of a warp add level widths one by one; lane 0 alone fences and
    counts the unit as done, and the lanes of the warp that finishes a pass sum
    the widths.  Shuffles and votes order no memory, so a __syncwarp stands
    between the additions and lane 0's fence, and between lane 0's second fence
    and the sums."""
    role = between(source("mc_cfg.cu"), "__device__ void warp_role", "__global__")
    before, rest = role.split("__threadfence();", 1)
    assert "__syncwarp();" in before[before.index("explore_unit_warp"):]
    assert before.rstrip().endswith("if (lane == 0) {")
    counted, combine = rest.split("cfg_epilogue_warp", 1)
    assert counted.index("units_done") < counted.index("__threadfence();") < counted.index("__syncwarp();")


def test_the_first_violating_level_is_read_by_one_lane():
    """The word with the least violating level falls while units run, and it
    decides whether a warp goes on to its next shuffle or vote.  Were it read
    by every lane, two lanes could see two values and part at a collective: one
    lane reads it, and the value it saw is shuffled to all before it decides
    anything."""
    units = [between(source("mc_cfg_wave.cuh"), "__device__ void explore_unit_wave", "template <class K, class C>"),
             between(source("mc_cfg.cu"), "__device__ uint32_t explore_unit_warp", "constexpr uint32_t kChainMaxP")]
    for text in units:
        reads = [m.start() for m in re.finditer(r"ld_relaxed_u32\(&ctrl->stop_c\)", text)]
        assert reads
        for at in reads:
            line = text[text.rindex("\n", 0, at) + 1:at]
            word = re.search(r"lane == 0\) (\w+) = $", line)
            assert word, line
            assert f"__shfl_sync(0xffffffffu, {word[1]}, 0)" in text
