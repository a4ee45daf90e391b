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


# kernels that a launch may start while the kernel before them still writes, and
# the names by which they read what that kernel writes
OVERLAPPED = [("agent_reg.cuh", "reg_body", r"x[rn]"), ("agent_reg.cuh", "reg32_body", r"x[rn]"),
              ("agent_xpose.cuh", "xpose_body", r"xr"), ("support.cu", "gather_chunk", r"v")]


def test_overlapped_kernels_read_live_data_by_plain_loads():
    """Read-only loads (__ldg, ld.global.nc, const restrict pointers) are for
    data that no one writes while the kernel is resident: under dependent
    launch the consensus image and the stack are not."""
    for name, body, var in OVERLAPPED:
        src = function(source(name), body)
        reads = re.findall(r"(\w+)\(%s(?: \+[^;]*?)?[,)]" % var, src)
        if name == "support.cu":   # the readout (mode 2) is launched without overlap
            src = re.sub(r"else if constexpr \(MODE == 2\)[^;]*;", "", src)
            reads = re.findall(r"(\w+)\(v \+ ", src)
        reads = [r for r in reads if r != "ld_live" and r != "ld_l2_hint"]
        assert not reads, (body, reads)
        assert not re.search(r"__restrict__\s+%s\b" % var, src), body
    for name, fn in (("pdl.cuh", "ld_live"), ("cache_hints.cuh", "ld_l2_hint")):
        asm = function(source(name), fn)
        assert "asm volatile" in asm and ".nc" not in asm
    # the loads of the next window are read-only ones only in the kernel that is
    # launched without overlap
    reg = source("agent_reg.cuh")
    assert re.search(r"if constexpr \(LIVE\) return ld_live\(p\)", function(reg, "ld_next"))
    assert "live ? agent_reg_kernel<N, true> : agent_reg_kernel<N, false>;" in reg and "pdl_launch(live, fn," in reg
    assert "reg_body<N, false>(a, wk.y" in reg
    # pdl_wait comes before the first of these reads
    for name, body, var in OVERLAPPED[:3]:
        src = function(source(name), body)
        assert src.index("pdl_wait()") < min(src.index(f"{f}(") for f in ("ld_live",) if f"{f}(" in src)
