"""The build compiles the walk objects that the dispatch reaches, and no others."""
import os
import re

from paper_1211_2293_gb300 import build


def test_walk_objects_are_reached():
    src = open(os.path.join(build.CSRC, "tc_walk.cu")).read()
    reached = {f"tc_walk_b{b}_t{t}" for b, t in re.findall(r"fn##_b(\d+)_t(\d+)\(", src)}
    assert reached == {obj for obj, _, _ in build.WALK_UNITS}
    assert {f"tc_walk_ws_t{t}" for t in re.findall(r"TC_WALK_WS_DECL\((\d+)\)", src)} == {
        obj for obj, _, _ in build.WALK_WS_UNITS}
