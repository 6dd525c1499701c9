"""Where the lanes of a warp hand simplex state to each other through memory, a warp barrier lies
between the store and the load: votes and shuffles order no memory.  (Read from the source: a
missing barrier is a race, which a run need not show.)"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1306_1122_gb300", "csrc")


def _code(name):
    src = open(os.path.join(CSRC, name)).read()
    return re.sub(r"/\*.*?\*/|//[^\n]*", "", src, flags=re.S)


def _between(src, first, last):
    i = src.index(first) + len(first)
    return src[i:src.index(last, i)]


def test_decided_steps_are_visible_to_the_lanes_that_form_trial_points():
    # decide(): a point's lane stores its vertices; then lanes per lambda read them
    assert "__syncwarp();" in _between(_code("solve_step.cuh"), "if (on) decide();", "SV(")


def test_values_are_visible_to_the_lanes_that_decide():
    # value lanes store their values; then the point's lane reads them
    src = _between(_code("solve_step.cuh"), "SD(a, D_REFS + s, og) = S[s];", "auto decide")
    assert "__syncwarp();" in src


def test_counts_are_read_before_points_are_added():
    # every lane reads the side's counts; then lanes add points to them
    src = _between(_code("search.cu"), "const int want =", "init_point<N>(")
    assert "__syncwarp();" in src
