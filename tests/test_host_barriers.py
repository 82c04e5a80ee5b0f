"""The trajectory step's stage kernel, read as text (no GPU): a scenario's status is read
and written by one warp of its block, which hands its verdict to the others over a
barrier that every thread reaches.  (A warp that read the status by itself could read it
after another warp had retired the scenario, and leave before the barrier.)"""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _body(src, name):
    """Text between the braces of kernel `name`."""
    at = src.index("{", src.index(name + "("))
    depth = 0
    for i in range(at, len(src)):
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        if depth == 0:
            return src[at + 1:i]
    raise AssertionError(name)


def test_stage_kernel_reads_the_status_in_one_warp():
    src = open(os.path.join(ROOT, "paper_2406_07048_gb300", "csrc", "oca_riccati.cu")).read()
    body = re.sub(r"//[^\n]*", "", _body(src, "k_traj_stage"))
    before, after = body.split("__syncthreads();", 1)
    assert not re.search(r"\breturn\b", before)
    assert not re.search(r"scen_status|stop_rule", after)
    # before the barrier, both only within the block that one warp runs
    head, warp0 = before.split("if (lane < 32)", 1)
    assert not re.search(r"scen_status|stop_rule", head)
    assert re.search(r"scen_status", warp0) and re.search(r"stop_rule", warp0)
