"""Rules of the CUDA programming model that no result shows: a kernel that breaks one may run
right for years, so they are read off the kernels' sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1306_2461_gb300", "csrc")


def code_of(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


SOURCES = sorted(n for n in os.listdir(CSRC) if n.endswith((".cu", ".cuh")))


@pytest.mark.parametrize("name", SOURCES)
def test_remote_shared_memory_between_cluster_barriers(name):
    # another block's shared memory is accessed after a cluster barrier (the block has started)
    # and before another one (it has not ended)
    for body in re.findall(r"__cluster_dims__.*?\n}\n", code_of(name), flags=re.S):
        barriers = [m.start() for m in re.finditer(r"barrier_wait\(\)|cluster\.sync\(\)", body)]
        for m in re.finditer(r"map_shared_rank", body):
            assert any(b < m.start() for b in barriers) and any(b > m.start() for b in barriers)
        assert len(re.findall(r"barrier_arrive\(\)", body)) == len(re.findall(r"barrier_wait\(\)", body))


@pytest.mark.parametrize("name", SOURCES)
def test_votes_name_lanes_that_arrive(name):
    # __activemask() gives whichever lanes happen to be converged: lanes may then hold different
    # masks for one vote, which is undefined. A vote or reduction names the whole warp, or the
    # lanes of a ballot of the whole warp.
    code = code_of(name)
    assert "__activemask" not in code
    masks = {"0xffffffffu"} | set(re.findall(r"(\w+) = __ballot_sync\(0xffffffffu,", code))
    for m in re.finditer(r"__(?:all|any|ballot|shfl\w*|reduce_\w+|match\w*)_sync\(([^,]*),", code):
        assert m.group(1).strip() in masks


def test_flow_modes_are_asked_of_mode_is():
    # a kernel's MODE may stand for two modes (FLOW_FIRST: a level's first iteration) or for any (-1);
    # compared as a number it matches neither, and a prefetch then warms nothing
    code = code_of("of_kernels.cuh")
    body = code[code.index("bool mode_is("):]
    body = code.replace(body[:body.index("\n}\n")], "")
    for m in re.finditer(r"\bmode == FLOW_\w+|\bMODE >= 0", body):
        line = body[body.rfind("\n", 0, m.start()) + 1:body.index("\n", m.end())]
        assert "a.mode" in line and "MODE >= 0" not in line, line
