"""Ordering rules of the simulation kernel that no run shows to be broken: they
are read off its source."""
import os
import re

from paper_2505_05286_gb300 import build as B


def _sim_body():
    """sim_body without its comments."""
    with open(os.path.join(B.CSRC, "hx_kernels.cu")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    start = text.index("void sim_body(")
    return text[start:text.index("\n}\n", start)]


def test_scratch_slices_reach_every_lane_before_their_first_use():
    """Lane 0 writes the warp's scratch pointers once: a barrier comes before any
    other lane reads one."""
    after = _sim_body().split("W->topk = a.topk + gw * a.topk_per_warp;")[1]
    assert "__syncwarp();" in after[:re.search(r"W->(arena|chains|topk)\b", after).start()]


def test_prefetches_end_before_the_kernel_does():
    """cp.async copies that nobody reads are waited for before the block exits."""
    body = _sim_body()
    assert "cp.async.ca" in body
    assert "cp.async.wait_all;" in body[body.rindex("__syncwarp();"):]
