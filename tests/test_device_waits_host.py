"""Checks of the kernels' waits and loads that can be made on the sources, with
no GPU: what must hold whatever the timing, and a GPU run would show only by
chance."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2111_14240_gb300", "csrc")


def source(name):
    """A file of csrc/ without its comments."""
    src = open(os.path.join(CSRC, name)).read()
    return re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", src), flags=re.S)


def function(src, name):
    """The body of the function `name`."""
    at = src.index("{", re.search(r"\b%s\(" % name, src).end())
    depth, i = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        i += 1
        if depth == 0:
            return src[at:i]


def test_register_sweep_lanes_agree_on_a_bounded_wait():
    """Warp-wide instructions follow every wait of the register sweeps, so the
    lanes vote on its outcome: no wait is taken by a lane for itself."""
    src = source("agent_reg.cuh")
    vote = function(src, "mbar_wait_warp")
    assert re.search(r"__all_sync\(0xffffffffu,\s*mbar_wait_bounded\(", vote)
    assert "mbar_wait_bounded" not in src.replace(vote, "")
    for body in ("reg_body", "reg32_body"):
        assert function(src, body).count("mbar_wait_warp(") == 2
    assert "mbar_try_wait" not in src
