"""A job of the layer team is not looked at after its last barrier.

The layer warp writes the job descriptor (LayerJob, in shared memory) for the team and goes on to its next job as soon as it has
passed the last barrier of the one before.  A thread of the team that still reads the descriptor then may see either job.  No run
shows such a read reliably, so the sources are looked at: in every function that works on a job, nothing of the job may be
named after the function's last barrier, and the loops that call them name it only after the barrier that hands it over.
"""
import os
import re

import pytest

from paper_2406_17276_b200 import build

JOB = re.compile(r"\bj\.\w|\bjob\.\w")


def _code(name):
    with open(os.path.join(build.CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _bodies(text):
    """(name, body) of the functions of `text` (braces matched)."""
    for m in re.finditer(r"__device__[^;{}]*?(\w+)\([^;{}]*\)\s*(?:const\s*)?\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i - 1]


def _job_functions():
    return [(n, b) for n, b in _bodies(_code("select.cuh")) if "s.job;" in b and "team_sync();" in b]


@pytest.mark.parametrize("name", ["select_layer_team", "select_running_team", "select_layer_team_big", "update_running", "update_running_staged"])
def test_nothing_of_the_job_is_read_after_the_last_barrier(name):
    bodies = [b for n, b in _job_functions() if n == name]
    assert len(bodies) == 1
    assert not JOB.findall(bodies[0].rsplit("team_sync();", 1)[1])


def test_every_job_function_is_looked_at():
    assert {n for n, _ in _job_functions()} == {"select_layer_team", "select_running_team", "select_layer_team_big", "update_running",
                                                "update_running_staged"}


def test_the_assistants_read_a_job_between_its_barriers():
    """In the assistants' loops each branch's first look at the job follows the barrier that hands it over, and what they call is
    one of the functions above, or ends with a barrier of its own."""
    loops = [b for n, b in _bodies(_code("opt_tree.cu")) if n == "layer_assist" and "team_sync();" in b]
    assert len(loops) == 2
    for body in loops:
        assert not JOB.findall(body.split("team_sync();", 1)[0])
        for line in body.split("\n"):
            if "pack_tree" in line:
                assert "team_sync();" in line.rsplit("job.", 1)[1]
