"""Memory comes from fmm_build_tree alone: no other call allocates (a call may be
made while another thread captures a graph, where allocations are refused)."""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1908_03121_gb300", "csrc")
ALLOC = re.compile(r"\bcuda(?:Malloc\w*|HostAlloc|HostRegister|StreamCreate\w*|EventCreate\w*)\s*\(")


def test_only_the_tree_build_allocates():
    for f in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        if f == "fmm_host.cpp":
            a = text.index("static int upload(T **dst")
            b = text.index('extern "C" {')
            assert len(ALLOC.findall(text[a:b])) >= 9
            text = text[:a] + text[b:]
        assert not ALLOC.findall(text), f
