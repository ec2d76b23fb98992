"""A process that ends with handles it never destroyed ends cleanly: each is
destroyed at exit as what it is."""
import os
import subprocess
import sys

import pytest

from conftest import ROOT

PROGRAM = """
import sys
sys.path.insert(0, {root!r})
from paper_2305_09130_gb300 import mc, pe_workloads as PW, workloads as W
keep = [mc.mc_model_create(W.c1(), allocator=None), mc.mc_pe_model_create(PW.pe_abstract(8, P=1), stream=0),
        mc.mc_batch_create([W.c1(), W.c2()], allocator=None), mc.mc_batch_create([W.c3()], allocator=None)]
{more}
print("end")
"""


def run(more):
    return subprocess.run([sys.executable, "-c", PROGRAM.format(root=ROOT, more=more)], cwd=ROOT, timeout=300,
                          capture_output=True, text=True, env=dict(os.environ, MALLOC_CHECK_="3"))


def test_handles_left_at_exit():
    r = run("")
    assert r.returncode == 0 and r.stdout == "end\n" and r.stderr == "", (r.returncode, r.stderr)


@pytest.mark.gpu
def test_handles_left_at_exit_after_queries(mc):
    r = run("""
assert mc.mc_count_states(keep[0]) > 0 and mc.mc_pe_count_states(keep[1]) > 0
assert mc.mc_batch_run(keep[2], [("min_time", None)] * 2)[0]["status"] == 0
keep.append(mc.mc_server_create(slots=4, pool_bytes=1 << 28))
mc.mc_server_submit(keep[-1], W.c1(), "min_time")
""")
    assert r.returncode == 0 and r.stdout == "end\n", (r.returncode, r.stderr)
