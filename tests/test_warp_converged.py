"""Source rules for warp-wide instructions: one that PTX wants executed by a whole
converged warp follows an instruction that brings the warp together, and its condition
is the same in every lane (a value that another warp may write is voted on first)."""

import os
import re

import paper_2205_00393_gb300

CSRC = os.path.join(os.path.dirname(paper_2205_00393_gb300.__file__), "csrc")


def _sources():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, name)) as f:
                yield name, re.sub(r"//[^\n]*", "", f.read())


def test_aligned_cluster_barriers_follow_a_syncwarp():
    for name, src in _sources():
        for m in re.finditer(r'asm volatile\("barrier\.cluster\.[^"]*\.aligned', src):
            assert src[:m.start()].rstrip().endswith("__syncwarp();"), name


def test_elections_do_not_depend_on_a_flag_of_another_warp():
    found = 0
    for name, src in _sources():
        for line in src.splitlines():
            if "elect_one()" in line and "bool elect_one" not in line:
                found += 1
                assert "abort_flag" not in line or "__any_sync(0xffffffffu, *abort_flag)" in line, (name, line.strip())
    assert found >= 4
